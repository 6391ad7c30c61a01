"""What a user of this framework has it do, as timed cases through its public entry points.

Kinds of case (the keys of a case besides its name):

* ``heff``: one projected-Hamiltonian application H.psi on device vectors
  (``apply_heff``), the call that an eigensolver of the user's own makes some
  hundred times per bond, on an environment that is kept: native FP64 or BF16
  slices (5 or 6 of them), operators on the device or streamed from pinned
  host memory (``resident_mb`` of them kept).
* ``heff_host``: the same from pinned host vectors (``apply_heff_host``), for
  a program that holds its wavefunction on the host.
* ``davidson``: the framework's own eigensolver from a start vector:
  creation (with the diagonal of H_eff), a number of iterations, eagerly or
  as a CUDA graph, and the Ritz vector.
* ``environment``: the operators of a window built from the integrals
  (block operators renormalised orbital by orbital on the GPU, operator
  slabs cut), its diagonal and one H.psi: what each new window costs before
  its eigensolver runs.

Sizes are bond dimensions D (kept multiplets per bond) and chain lengths L
of the configurations, tests and benchmark of this repository, and other
values between them.
"""
import math

import numpy as np
import torch

import paper_2309_16724_gb300 as P
import synth
from paper_2309_16724_gb300 import workload


def _case(kind, L, N, twoS, D, prec="split", slices=5, site="orbital", resident_mb=0, budget_mb=0, steps=0,
          graph=False, name=None):
    c = dict(kind=kind, site=site, L=L, N=N, twoS=twoS, D=D, prec=prec, slices=slices, resident_mb=resident_mb,
             budget_mb=budget_mb, steps=steps, graph=graph)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call: a spin chain, every block tiny; launches and latency count
        _case("heff", 12, 12, 0, 32, prec="fp64", site="spin", name="heff-fp64-spin-L12-D32"),
        # a small molecule's window near the chain's end: blocks of 5 to 30
        # rows, split path, most of the chip idle
        _case("heff", 12, 12, 0, 100, name="heff-split-L12-D100"),
        # the double-precision reference path on an ordinary window
        _case("heff", 16, 16, 0, 512, prec="fp64", name="heff-fp64-L16-D512"),
        # an ordinary window on the path that sweeps run on
        _case("heff", 16, 16, 0, 512, name="heff-split-L16-D512"),
        # an open-shell target (S = 1/2), odd chain and ragged sectors, with
        # the six slices of a tightly converged final sweep
        _case("heff", 19, 19, 1, 700, slices=6, name="heff-split6-L19-S1/2-D700"),
        # a wide window: large bond dimension on a medium chain
        _case("heff", 20, 20, 0, 1536, name="heff-split-L20-D1536"),
        # the largest: long chain, large bond dimension, seconds of CPU time per call
        _case("heff", 32, 32, 0, 2048, name="heff-split-L32-D2048"),
        # operators kept in host memory and streamed by term chunks
        _case("heff", 18, 18, 0, 900, resident_mb=100, budget_mb=256, name="heff-split-streamed-L18-D900"),
        # the eigensolver on an ordinary window, as the sweep runs it
        _case("davidson", 16, 16, 0, 512, steps=6, name="davidson-split-L16-D512"),
        # the eigensolver on a small open-shell window in double precision,
        # one iteration a graph launch
        _case("davidson", 11, 11, 1, 72, prec="fp64", steps=16, graph=True, name="davidson-fp64-graph-L11-S1/2-D72"),
        # a new window from the integrals: renormalisation, slabs, first H.psi
        _case("environment", 12, 12, 0, 150, name="environment-L12-D150"),
    ]


# cost of a case, for keeping drawn cases below the largest listed one:
# flops of H.psi grow about as D^3 L^2 (8.1e12 at L = 32, D = 2048, S = 0)
def _gflop(L, D, twoS):
    return 8100.0 * (D / 2048.0) ** 3 * (L / 32.0) ** 2 * (2.0 if twoS else 1.0)


def draw(rng):
    kind = rng.choice(["heff", "heff", "heff", "heff", "heff_host", "davidson", "environment"])
    twoS = rng.choice([0, 0, 0, 1, 2])
    if kind == "environment":
        L = rng.randint(7, 12)
        D = int(round(math.exp(rng.uniform(math.log(12), math.log(160)))))
        return _case(kind, L, L - (L - twoS) % 2, twoS, D)
    prec = rng.choice(["split", "split", "split", "fp64"])
    if rng.random() < 0.08:
        L = rng.randint(8, 14)
        D = rng.randint(6, 40)
        return _case("heff", L, L, L % 2, D, prec=prec, site="spin")
    if kind == "davidson":
        limit, hi = 100.0, 700
    elif prec == "fp64":
        limit, hi = 200.0, 900
    else:
        limit, hi = 6000.0, 2000
    while True:
        L = rng.randint(8, 32)
        D = int(round(math.exp(rng.uniform(math.log(12), math.log(hi)))))
        if _gflop(L, D, twoS) <= limit:
            break
    N = L - (L - twoS) % 2
    kw = {}
    if kind == "davidson":
        kw = dict(steps=rng.randint(3, 8), graph=rng.random() < 0.3)
    elif kind == "heff" and rng.random() < 0.2:
        kw = dict(resident_mb=rng.choice([20, 50, 200]), budget_mb=rng.choice([64, 128, 512]))
    return _case(kind, L, N, twoS, D, prec=prec, slices=rng.choice([5, 5, 5, 6]), **kw)


def _config(case, seed):
    site = synth.SPIN_HALF if case["site"] == "spin" else synth.SPATIAL_ORBITAL
    return synth.Config("case", site, case["L"], case["N"], case["twoS"], case["D"], int(seed))


def _env_options(case):
    return dict(prepare_split=case["prec"] == "split", n_slices=case["slices"],
                t_budget_bytes=case["budget_mb"] << 20, resident_bytes=case["resident_mb"] << 20)


def _psi(n, seed):
    """A normalised Gaussian wavefunction, made on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    return x / torch.linalg.vector_norm(x)


def _first_order(heff, diag):
    """The start vector of an eigensolver: the basis state of lowest diagonal
    element and its first-order correction.  Its energy lies below every
    diagonal element, so the iterations are those of a sound start."""
    i = int(diag.argmin())
    e = torch.zeros_like(diag)
    e[i] = 1.0
    h = heff(e)
    h[i] = 0.0
    x = e - h / (diag - diag[i] + 0.5)
    return x / torch.linalg.vector_norm(x)


def prepare(case, seed):
    ctx = P.Context(0, stream=torch.cuda.current_stream())
    cfg = _config(case, seed)
    s = dict(case=case, ctx=ctx, cfg=cfg, prec=P.SU2_SPLIT_BF16 if case["prec"] == "split" else P.SU2_FP64)
    if case["kind"] == "environment":
        s["h"], s["eri"] = synth.integrals(cfg.L, cfg.seed)
        s["left"], s["right"] = workload.chains(cfg)
        n = P.Sectors(ctx, s["left"][-1], s["right"][-1], cfg.site_kind, cfg.N, cfg.twoS).psi_len
    else:
        s["sec"], s["env"] = workload.build(ctx, cfg, **_env_options(case))
        n = s["sec"].psi_len
    if case["kind"] == "davidson":
        diag = torch.empty(n, dtype=torch.float64, device="cuda")
        P.diag_heff(ctx, s["env"], diag)

        def heff(v):
            w = torch.empty_like(v)
            P.apply_heff(ctx, s["env"], v, w, P.SU2_FP64)
            return w

        s["x"] = _first_order(heff, diag)
    else:
        s["x"] = _psi(n, seed + 100)
    if case["kind"] == "heff_host":
        s["x"] = s["x"].cpu().pin_memory()
        s["y"] = torch.empty(n, dtype=torch.float64).pin_memory()
    else:
        s["y"] = torch.empty_like(s["x"])
    if case["kind"] == "environment":
        s["diag"] = torch.empty_like(s["x"])
    return s


def run(s):
    kind, ctx, cfg = s["case"]["kind"], s["ctx"], s["cfg"]
    if kind == "heff":
        P.apply_heff(ctx, s["env"], s["x"], s["y"], s["prec"])
        return s["y"]
    if kind == "heff_host":
        P.apply_heff_host(ctx, s["env"], s["x"], s["y"], s["prec"])
        return s["y"]
    if kind == "davidson":
        # a fixed number of iterations: tol is out of reach on purpose
        d = P.Davidson(ctx, s["env"], s["x"], tol=1e-13, prec=s["prec"], use_graph=s["case"]["graph"])
        steps = [d.step() for _ in range(s["case"]["steps"])]
        d.vector(s["y"])
        d.close()
        return {"theta": np.array([t for t, _ in steps]), "residual": np.array([r for _, r in steps]), "vector": s["y"]}
    sec = P.Sectors(ctx, s["left"][-1], s["right"][-1], cfg.site_kind, cfg.N, cfg.twoS)
    env = P.Environment(ctx, sec, P.SU2_MODEL_AB_INITIO, s["left"], s["right"], n_left=cfg.n_left,
                        n_right=cfg.n_right, seed=cfg.seed, h=s["h"], eri=s["eri"], **_env_options(s["case"]))
    P.diag_heff(ctx, env, s["diag"])
    P.apply_heff(ctx, env, s["x"], s["y"], s["prec"])
    env.close()
    return {"diagonal": s["diag"], "heff": s["y"]}


def work(case):
    """The sector products and operators of one H.psi, times the number of
    H.psi of a pass; a Davidson iteration also reads its subspace."""
    ctx = P.Context(0, stream=torch.cuda.current_stream())
    cfg = _config(case, 1)
    kw = dict(model=P.SU2_MODEL_AB_INITIO) if case["kind"] == "environment" else {}
    sec, env = workload.build(ctx, cfg, **kw)
    n, ops, flops = 8.0 * sec.psi_len, env.info["env_bytes"], env.info["flops_su2"]
    env.close()
    if case["kind"] == "davidson":
        k = case["steps"]
        # per iteration: one H.psi; V and A V read for the Ritz vector, V
        # twice per Gram-Schmidt pass and once for the projected matrix
        return {"bytes": k * ops + n * sum(2 + 7 * (i + 1) for i in range(k)),
                "flops": k * flops + 2.0 * sec.psi_len * sum(7 * (i + 1) for i in range(k))}
    if case["kind"] == "environment":
        return {"bytes": 2 * ops + 3 * n, "flops": flops + env.info["renorm_flops"]}
    return {"bytes": ops + 2 * n, "flops": flops}


class _Heff:
    """F = sum_t v_t A_t E_t D_t^T (the sum over the sector-task table of the
    environment, its coefficients and operator blocks read back as data) in
    64-bit torch products."""

    def __init__(self, sec, env):
        rows, v = env.tasks()
        ta, td, _, _ = env.terms()
        blocks = {0: {}, 1: {}}

        def op(side, o, qo, qi, m, k):
            key = (o, qo, qi)
            if key not in blocks[side]:
                blocks[side][key] = torch.from_numpy(np.ascontiguousarray(env.operator_block(side, o, qo, qi, m, k))).cuda()
            return blocks[side][key]

        B = sec.blocks
        self.n = sec.psi_len
        self.shape = [(b[6], b[7], b[8]) for b in B]
        self.plan = []
        for (f, term, e, ao, ai, bo, bi, flags), vt in zip(rows.tolist(), v.tolist()):
            A = None if flags & 1 else op(0, int(ta[term]), ao, ai, B[f][6], B[e][6])
            D = None if flags & 2 else op(1, int(td[term]), bo, bi, B[f][7], B[e][7])
            self.plan.append((f, e, vt, A, D, None if D is None else (int(td[term]), bo, bi, e)))

    def __call__(self, x):
        E = [x[o:o + m * n].view(n, m).T for m, n, o in self.shape]
        out = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        F = [out[o:o + m * n].view(n, m).T for m, n, o in self.shape]
        T = {}
        for f, e, v, A, D, key in self.plan:
            if D is None:
                t = E[e]
            else:
                t = T.get(key)
                if t is None:
                    t = T[key] = E[e] @ D.T
            if A is None:
                F[f].add_(t, alpha=v)
            else:
                F[f].addmm_(A, t, alpha=v)
        return out

    def diagonal(self):
        out = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        F = [out[o:o + m * n].view(n, m).T for m, n, o in self.shape]
        for f, e, v, A, D, _ in self.plan:
            if e == f:
                a = torch.ones(self.shape[f][0], dtype=torch.float64, device="cuda") if A is None else A.diagonal()
                d = torch.ones(self.shape[f][1], dtype=torch.float64, device="cuda") if D is None else D.diagonal()
                F[f].add_(torch.outer(a, d), alpha=v)
        return out


def _davidson(H, x, steps):
    """Fixed number of Davidson iterations (no restart within them): lowest
    Ritz value, residual norm and Ritz vector of each subspace, the
    correction r / (diag - theta) orthogonalised twice."""
    diag = H.diagonal()
    V, W, theta, res = [x / torch.linalg.vector_norm(x)], [], [], []
    for _ in range(steps):
        W.append(H(V[-1]))
        Vm, Wm = torch.stack(V), torch.stack(W)
        G = Vm @ Wm.T
        w, Y = torch.linalg.eigh(0.5 * (G + G.T))
        u, Au = Y[:, 0] @ Vm, Y[:, 0] @ Wm
        r = Au - w[0] * u
        theta.append(float(w[0]))
        res.append(float(torch.linalg.vector_norm(r)))
        d = diag - w[0]
        t = r / torch.where(d.abs() < 1e-12, torch.where(d >= 0, 1e-12, -1e-12).to(d), d)
        for _ in range(2):
            t = t - (Vm @ t) @ Vm
        V.append(t / torch.linalg.vector_norm(t))
    # the library's sign: the component of largest magnitude is positive
    u = u / torch.linalg.vector_norm(u)
    return theta, res, u * torch.sign(u[u.abs().argmax()])


def exact(case, seed):
    ctx = P.Context(0, stream=torch.cuda.current_stream())
    cfg = _config(case, seed)
    if _gflop(cfg.L, cfg.D, cfg.twoS) * max(1, case["steps"]) > 600.0 and case["site"] == "orbital":
        return None
    kw = dict(model=P.SU2_MODEL_AB_INITIO) if case["kind"] == "environment" else {}
    sec, env = workload.build(ctx, cfg, **kw)
    H = _Heff(sec, env)
    if case["kind"] == "davidson":
        theta, res, u = _davidson(H, _first_order(H, H.diagonal()), case["steps"])
        return {"theta": np.array(theta), "residual": np.array(res), "vector": u}
    x = _psi(sec.psi_len, seed + 100)
    if case["kind"] == "environment":
        return {"diagonal": H.diagonal(), "heff": H(x)}
    return H(x).cpu() if case["kind"] == "heff_host" else H(x)

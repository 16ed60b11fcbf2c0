"""The work that a user of this library has it do, as cases that can be timed.

Each case is one pass through the public binding (paper_2603_12550_gb300.vds):
full-order time steps and evaluations, the bandwidth rule, batched ensembles,
the POD build, the two reduced steps, a training burst of the score network
and the convection between grid nodes.  Sizes are those of this repository's
workloads (inputs.WORKLOADS, the benchmark, the tests); draw() spreads them
over the ranges between.  Inputs are drawn on the GPU from the seed alone.
exact() is the same result in 64 bits, in plain torch.
"""
import math

import numpy as np
import torch

from paper_2603_12550_gb300 import vds

DEV = "cuda"
KBT, ZETA = 1.0, 4.0
FENE_B = 50.0

# D = nb * s: the chains that the pair passes are built for
CHAINS = [(1, 2), (1, 3), (2, 2), (2, 3), (4, 2), (3, 3), (5, 2), (4, 3), (7, 2), (5, 3), (8, 2)]
# ... and those of the batched form
BATCH_CHAINS = [(1, 2), (1, 3), (2, 2), (2, 3), (4, 2), (3, 3), (4, 3)]


def listed():
    return [
        # the headline workload: explicit steps of 65536 four-bead chains in shear
        dict(name="explicit_chain4_65536", kind="explicit", N=65536, nb=3, s=3, spring=0, strain=0.5, dt=0.005,
             steps=2),
        # the paper's own size (P = 1000 four-bead chains, thousands of explicit steps at dt = 1e-3)
        dict(name="explicit_chain4_1000", kind="explicit", N=1000, nb=3, s=3, spring=0, strain=0.5, dt=0.001,
             steps=50),
        # the 3D dumbbell cloud of the rheology runs
        dict(name="explicit_dumbbell3d_16384", kind="explicit", N=16384, nb=1, s=3, spring=0, strain=0.0, dt=0.005,
             steps=10),
        # the 2D dumbbell, implicit Euler by the minimiser: small and launch bound
        dict(name="implicit_dumbbell2d_512", kind="implicit", N=512, nb=1, s=2, spring=0, strain=0.5, h=0.3, dt=0.01,
             steps=5),
        # energy, gradient and density of a FENE cloud of ragged size (a user's own integrator)
        dict(name="evaluate_fene3_10007", kind="evaluate", N=10007, nb=2, s=3, spring=1, strain=0.5),
        # kernel bandwidth by the median rule, at the start of every run
        dict(name="bandwidth_chain4_65536", kind="bandwidth", N=65536, nb=3, s=3, strain=0.0),
        # micro-macro coupling: one implicit step of uneven ensembles of three-bead chains
        dict(name="batch_implicit_96", kind="batch", E=96, lo=10.0, hi=14.0, nb=2, s=3, scheme=1, steps=1),
        # convection of those ensembles between the nodes of an 8 x 8 x 8 grid
        dict(name="convect_512", kind="convect", nx=8, ny=8, nz=8, M=98304, bc=0),
        # POD basis from the 200 snapshots of a full-order run
        dict(name="pod_build_600", kind="pod", N=65536, nb=3, s=3, snaps=200, r=6),
        # the frozen reduced step with its X^B refresh every 60 steps
        dict(name="frozen_chain4_65536", kind="frozen", N=65536, nb=3, s=3, r=10, steps=120, refresh=60, strain=0.5),
        # the score surrogate in the reduced step with its exact check every 20 steps
        dict(name="surrogate_chain4_262144", kind="surrogate", N=262144, nb=3, s=3, r=6, steps=40, check=20,
             strain=0.5),
        # a burst of training steps of the score network, then its weights
        dict(name="train_8192", kind="train", M=8192, pool=131072, nb=3, s=3, steps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["explicit", "explicit", "explicit", "implicit", "evaluate", "evaluate", "bandwidth", "batch",
                       "convect", "pod", "frozen", "surrogate", "train"])
    nb, s = rng.choice(CHAINS)
    if kind == "explicit":
        # from the 2D dumbbell's cloud to the headline's; more steps where a step is short
        if rng.random() < 0.4:  # the chains of the paper and of the benchmark
            nb, s = rng.choice([(1, 3), (2, 3), (3, 3)])
        N = _log(rng, 500, 65536 if nb * s <= 9 else 40000)
        return dict(kind=kind, N=N, nb=nb, s=s, spring=rng.choice([0, 0, 1]), strain=round(rng.uniform(0.0, 1.5), 2),
                    dt=rng.choice([0.001, 0.005]), steps=2 if N > 20000 else 10 if N > 4000 else 50)
    if kind == "implicit":
        nb, s = rng.choice([(1, 2), (1, 3), (2, 3), (3, 3)])
        N = _log(rng, 500, 16384)
        return dict(kind=kind, N=N, nb=nb, s=s, spring=0, strain=round(rng.uniform(0.0, 1.0), 2),
                    h=0.3 if nb * s == 2 else 0.0, dt=rng.choice([0.005, 0.01]), steps=3)
    if kind == "evaluate":
        return dict(kind=kind, N=_log(rng, 300, 50000 if nb * s <= 9 else 30000), nb=nb, s=s,
                    spring=rng.choice([0, 1]), strain=round(rng.uniform(0.0, 1.5), 2))
    if kind == "bandwidth":
        return dict(kind=kind, N=_log(rng, 500, 65536), nb=nb, s=s, strain=round(rng.uniform(0.0, 1.5), 2))
    if kind == "batch":
        nb, s = rng.choice(BATCH_CHAINS)
        return dict(kind=kind, E=_log(rng, 16, 128), lo=rng.choice([8.0, 9.0, 10.0]), hi=rng.choice([11.0, 12.0, 13.0]),
                    nb=nb, s=s, scheme=rng.choice([0, 1]), steps=1)
    if kind == "convect":
        return dict(kind=kind, nx=rng.randint(1, 12), ny=rng.randint(1, 8), nz=rng.choice([1, 1, 4, 5]),
                    M=_log(rng, 900, 98304), bc=rng.choice([0, 1]))
    if kind == "pod":
        nb, s = rng.choice([(1, 3), (2, 3), (3, 3)])
        return dict(kind=kind, N=_log(rng, 1000, 65536), nb=nb, s=s, snaps=rng.randint(20, 600 // nb // 2),
                    r=rng.randint(3, 6))
    if kind == "frozen":
        nb, s = rng.choice([(1, 3), (2, 3), (3, 3)])
        return dict(kind=kind, N=_log(rng, 1000, 65536), nb=nb, s=s, r=rng.randint(4, 20), steps=120, refresh=60,
                    strain=round(rng.uniform(0.0, 1.0), 2))
    if kind == "surrogate":
        nb, s = rng.choice([(2, 3), (3, 3)])
        return dict(kind=kind, N=_log(rng, 20000, 200000), nb=nb, s=s, r=rng.randint(4, 10), steps=40,
                    check=rng.choice([20, 40]), strain=round(rng.uniform(0.0, 1.0), 2))
    nb, s = rng.choice([(1, 3), (2, 3), (3, 3)])
    return dict(kind=kind, M=128 * rng.randint(8, 64), pool=_log(rng, 10000, 262144), nb=nb, s=s, steps=16)


# ------------------------------------------------------------------ inputs

def _shear(s, rate=1.0):
    k = np.zeros((s, s))
    k[0, 1] = rate
    return k


def _bandwidth(N, D):
    """The median rule's h for N equilibrium particles (|x - y|^2 / 2 is chi-squared of D)."""
    return math.sqrt(2.0 * D * (1.0 - 2.0 / (9.0 * D)) ** 3 / (2.0 * math.log(N)))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _cloud(N, nb, s, strain, gen, spring=0):
    """An equilibrium cloud carried through a shear strain; FENE bonds stay inside their domain."""
    q = torch.randn((N, nb, s), device=DEV, generator=gen)
    q[..., 0] += strain * q[..., 1]
    if spring == 1:
        n2 = (q * q).sum(-1, keepdim=True)
        q *= torch.sqrt((0.8 * FENE_B) / n2.clamp(min=0.8 * FENE_B))
    return q.reshape(N, nb * s).contiguous()


def _params(case, scheme=0):
    D = case["nb"] * case["s"]
    h = case.get("h") or _bandwidth(max(case["N"], 3), D)
    return vds.params(case["nb"], case["s"], H=1.0, kBT=KBT, zeta=ZETA, h=h, dt=case.get("dt", 0.005),
                      kappa=_shear(case["s"]), spring=case.get("spring", 0), b=FENE_B, tol=1e-6, jfloor=1e-9,
                      scheme=scheme)


def _snapshots(case, gen):
    """Snapshots like a full-order run's: shear that saturates, relaxing bonds, and weaker nonlinear modes
    that fade at their own rates; one row per (snapshot, bond)."""
    N, nb, s, S = case["N"], case["nb"], case["s"], case["snaps"]
    q0 = torch.randn((N, nb, s), device=DEV, generator=gen)
    modes = [torch.tanh(q0.reshape(N, nb * s) @ torch.randn((nb * s, nb * s), device=DEV, generator=gen) * 0.5)
             .reshape(N, nb, s) for _ in range(8)]
    X = torch.empty((S * nb, N * s), device=DEV)
    for l in range(S):
        t = 5.0 * (l + 1) / S
        q = (1.0 + 0.1 * math.exp(-t)) * q0
        q[..., 0] += (1.0 - math.exp(-0.5 * t)) * 1.5 * q0[..., 1]
        for m, f in enumerate(modes):
            q = q + 0.3 * 2.0 ** -(m + 1) * (math.exp(-0.3 * (m + 1) * t) - 0.2 * math.cos((m + 1) * t)) * f
        X[l * nb:(l + 1) * nb] = q.transpose(0, 1).reshape(nb, N * s)
    return X


def _reduced(case, gen):
    """An orthonormal basis that holds the cloud's bonds and smooth functions of them, and the cloud's coordinates."""
    N, nb, s, r = case["N"], case["nb"], case["s"], case["r"]
    q = _cloud(N, nb, s, case["strain"], gen).reshape(N, nb, s)
    cols = [q[:, k, :].reshape(-1) for k in range(nb)]
    while len(cols) < r:
        W = torch.randn((nb, nb), device=DEV, generator=gen)
        cols.append(torch.tanh(torch.einsum("nka,kj->nja", q, W)[:, 0, :]).reshape(-1))
    phi = torch.linalg.qr(torch.stack(cols[:r], 1).double())[0].float().contiguous()
    P = torch.stack([phi.double().T @ q[:, k, :].reshape(-1).double() for k in range(nb)], 1).float().contiguous()
    return phi, P


def _score_layers(D, gen):
    """A network near the score of the sheared cloud, s(x) = -0.6 x: SiLU units in pairs of opposite sign carry x
    through (silu(z) - silu(-z) = z), the others carry small random features."""
    Wd = 256
    n = 2 * D
    eye = torch.eye(D, device=DEV)
    pair = torch.cat([eye, -eye])
    mk = lambda o, i, sc: sc * torch.randn((o, i), device=DEV, generator=gen) / math.sqrt(i)  # noqa: E731
    W1, W2, W3, W4 = mk(Wd, D, 1.0), mk(Wd, Wd, 1.0), mk(Wd, Wd, 1.0), mk(D, Wd, 0.02)
    W1[:n] = pair
    for W in (W2, W3):
        W[:n] = 0.0
        W[:n, :n] = pair @ pair.T
    W4[:, :n] = -0.6 * pair.T
    z = lambda k: np.zeros(k, dtype=np.float32)  # noqa: E731
    return [(W.cpu().numpy().astype(np.float32), z(W.shape[0])) for W in (W1, W2, W3, W4)]


def _train_layers(D, seed):
    rng = np.random.default_rng(int(seed))
    w = (D, 256, 256, 256, D)
    return [((rng.standard_normal((o, i)) / math.sqrt(i)).astype(np.float32), np.zeros(o, dtype=np.float32))
            for i, o in zip(w[:-1], w[1:])]


def _train_draws(case, gen):
    D = case["nb"] * case["s"]
    x = _cloud(case["pool"], case["nb"], case["s"], 0.5, gen)
    rows = torch.randint(0, case["pool"], (case["steps"], case["M"]), device=DEV, generator=gen, dtype=torch.int32)
    eps = torch.randn((case["steps"], case["M"], D), device=DEV, generator=gen)
    return x, rows, eps, _bandwidth(case["pool"], D)


def _batch_sizes(case, seed):
    rng = np.random.default_rng(int(seed) % 1000)
    sizes = np.rint(2.0 ** np.linspace(case["lo"], case["hi"], case["E"])).astype(np.int64)
    return rng.permutation(sizes), 10.0 ** rng.uniform(-1.0, 1.0, case["E"])


# --------------------------------------------------------------- the passes

_ctx = None


def _context():
    """One context for the whole program, as a program has it."""
    global _ctx
    if _ctx is None:
        _ctx = vds.Context(0)
    return _ctx


def prepare(case, seed):
    kind, gen, ctx = case["kind"], _gen(seed), _context()
    st = dict(case=case, ctx=ctx)
    if kind == "explicit":
        st.update(q=_cloud(case["N"], case["nb"], case["s"], case["strain"], gen, case["spring"]), p=_params(case))
    elif kind == "implicit":
        q0 = _cloud(case["N"], case["nb"], case["s"], case["strain"], gen)
        st.update(q0=q0, q=torch.empty_like(q0), p=_params(case, scheme=1))
    elif kind == "evaluate":
        q = _cloud(case["N"], case["nb"], case["s"], case["strain"], gen, case["spring"])
        st.update(q=q, p=_params(case), g=torch.empty_like(q), rho=torch.empty(case["N"], device=DEV))
    elif kind == "bandwidth":
        st.update(q=_cloud(case["N"], case["nb"], case["s"], case["strain"], gen))
    elif kind == "batch":
        sizes, rates = _batch_sizes(case, seed)
        D = case["nb"] * case["s"]
        h = np.array([_bandwidth(int(n), D) for n in sizes])
        kap = np.stack([_shear(case["s"], r) for r in rates])
        p = vds.params(case["nb"], case["s"], kBT=KBT, zeta=ZETA, dt=0.005, scheme=case["scheme"], tol=1e-6,
                       jfloor=1e-9)
        q0 = _cloud(int(sizes.sum()), case["nb"], case["s"], 0.0, gen)
        st.update(q0=q0, q=torch.empty_like(q0), batch=vds.Batch(ctx, sizes, D, p, h, kap))
    elif kind == "convect":
        G = case["nx"] * case["ny"] * case["nz"]
        q = torch.randn((G, case["M"]), device=DEV, generator=gen)
        st.update(q=q, out=torch.empty_like(q), u=torch.randn((G, 3), device=DEV, generator=gen) * 0.5)
    elif kind == "pod":
        st.update(X=_snapshots(case, gen))
    elif kind == "frozen":
        phi, P = _reduced(case, gen)
        st.update(P=P, p=_params(case), basis=ctx.pod_load(phi, case["s"], _shear(case["s"])))
    elif kind == "surrogate":
        phi, P = _reduced(case, gen)
        D = case["nb"] * case["s"]
        st.update(P=P, p=_params(case), basis=ctx.pod_load(phi, case["s"], _shear(case["s"])),
                  net=vds.Score(ctx, D, _score_layers(D, gen)))
    elif kind == "train":
        x, rows, eps, sigma = _train_draws(case, gen)
        D = case["nb"] * case["s"]
        st.update(x=x, rows=rows, eps=eps, sigma=sigma, net=vds.Score(ctx, D, _train_layers(D, seed)))
    else:
        raise ValueError(kind)
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "explicit":  # in place, as a run goes on
        ctx.vds_step(st["q"], st["p"], case["steps"])
        return st["q"]
    if kind == "implicit":  # short runs from one start, as a study of step sizes or rates makes them
        st["q"].copy_(st["q0"])
        ctx.vds_step(st["q"], st["p"], case["steps"])
        return st["q"]
    if kind == "evaluate":
        E = ctx.vds_energy_grad(st["q"], st["p"], g=st["g"], rho=st["rho"])
        return E, st["g"], st["rho"]
    if kind == "bandwidth":
        return ctx.vds_bandwidth(st["q"], 0)
    if kind == "batch":
        st["q"].copy_(st["q0"])
        st["batch"].step(st["q"], case["steps"])
        return st["q"]
    if kind == "convect":
        ctx.vds_convect(st["q"], st["out"], (case["nx"], case["ny"], case["nz"]), st["u"], (0.5, 0.5, 0.5), 0.01,
                        case["bc"])
        return st["out"]
    if kind == "pod":
        s, X = case["s"], st["X"]
        basis, r = ctx.pod_build(X, case["N"] * s, X.shape[0], s, r_fixed=case["r"], kappa=_shear(s))
        res = dict(r=r, lam=basis.eigenvalues(), phi=basis.phi())
        basis.free()
        return res
    if kind == "frozen":
        ctx.pod_step(st["basis"], st["P"], case["N"], case["nb"] * case["s"], st["p"], nsteps=case["steps"],
                     refresh_every=case["refresh"], mode=2)
        return st["P"]
    if kind == "surrogate":
        err, fell_back = ctx.pod_step_score(st["basis"], st["net"], st["P"], case["N"], case["nb"] * case["s"],
                                            st["p"], nsteps=case["steps"], check_every=case["check"], check_n=4096,
                                            check_tol=0.9)
        return dict(P=st["P"], err=err, fell_back=fell_back)
    for k in range(case["steps"]):
        st["net"].train_step(st["x"], st["eps"][k], st["sigma"], 1e-3, want_loss=False, rows=st["rows"][k])
    return st["net"].params()


def work(case):
    kind = case["kind"]
    N, D = case.get("N", 0), case.get("nb", 0) * case.get("s", 0)
    pairs = 0.5 * N * N  # unordered; a kernel value is symmetric
    dens, grad = pairs * (3 * D + 3), pairs * (7 * D + 3)
    if kind == "explicit":
        return dict(bytes=8.0 * N * D, flops=case["steps"] * (dens + grad))
    if kind == "implicit":  # two gradients and two line-search densities a step
        return dict(bytes=8.0 * N * D, flops=case["steps"] * 2.0 * (dens + grad))
    if kind == "evaluate":
        return dict(bytes=4.0 * N * (2 * D + 1), flops=dens + grad)
    if kind == "bandwidth":
        return dict(bytes=4.0 * N * D, flops=pairs * 3 * D)
    if kind == "batch":
        sizes, _ = _batch_sizes(case, 0)
        pairs = 0.5 * float((sizes.astype(np.float64) ** 2).sum())
        per = pairs * (10 * D + 6) * (2.0 if case["scheme"] == 1 else 1.0)
        return dict(bytes=8.0 * float(sizes.sum()) * D, flops=case["steps"] * per)
    if kind == "convect":
        n = float(case["nx"] * case["ny"] * case["nz"]) * case["M"]
        return dict(bytes=8.0 * n, flops=8.0 * n)
    if kind == "pod":
        rows, M = float(N) * case["s"], case["snaps"] * case["nb"]
        return dict(bytes=4.0 * rows * M, flops=rows * M * (M + 1) + 4.0 * M ** 3)
    if kind == "frozen":
        r, s = case["r"], case["s"]
        n = -(-case["steps"] // case["refresh"])
        return dict(bytes=4.0 * N * s * r, flops=n * (dens + pairs * (3 * D + 1) + 2.0 * N * N * (2 * s * r + 1)))
    if kind == "surrogate":
        net = 2.0 * N * (2 * D * 256 + 2 * 256 * 256)
        n = -(-case["steps"] // case["check"])
        return dict(bytes=4.0 * N * case["s"] * case["r"], flops=case["steps"] * net + n * dens)
    per = 6.0 * case["M"] * (2 * D * 256 + 2 * 256 * 256)
    return dict(bytes=4.0 * case["steps"] * case["M"] * (2 * D + 1), flops=case["steps"] * per)


# ------------------------------------------------------------- in 64 bits

def _rows64(x, f):
    """f(rows, kernel-ready squared distances) over blocks of rows."""
    N = x.shape[0]
    n2 = (x * x).sum(1)
    B = max(1, min(N, (1 << 27) // N))
    for a in range(0, N, B):
        r2 = (n2[a:a + B, None] + n2[None, :] - 2.0 * (x[a:a + B] @ x.T)).clamp_(min=0.0)
        f(slice(a, min(N, a + B)), r2)


def _pairs64(x, h):
    """rho and the entropy gradient S."""
    N, D = x.shape
    rho = torch.empty(N, dtype=torch.float64, device=DEV)
    c = -0.5 / (h * h)

    def first(sl, r2):
        rho[sl] = r2.mul_(c).exp_().sum(1)
    _rows64(x, first)
    w = 1.0 / rho
    R = torch.cat([w[:, None], x, w[:, None] * x], 1)
    S = torch.empty_like(x)

    def second(sl, r2):
        V = r2.mul_(c).exp_() @ R
        S[sl] = -(x[sl] * (1.0 + V[:, :1]) - (w[sl, None] * V[:, 1:D + 1] + V[:, D + 1:])) / (h * h)
    _rows64(x, second)
    return rho, S


def _rouse(nb):
    return (2.0 * torch.eye(nb) - torch.diag(torch.ones(nb - 1), 1) - torch.diag(torch.ones(nb - 1), -1)
            ).double().to(DEV)


def _force(x, nb, s, spring):
    q = x.reshape(-1, nb, s)
    if spring == 0:
        return x
    return (q / (1.0 - (q * q).sum(-1, keepdim=True) / FENE_B)).reshape(x.shape)


def _flow(x, nb, s, kap):
    return torch.einsum("ab,nkb->nka", kap, x.reshape(-1, nb, s)).reshape(x.shape)


def _rouse_mul(g, nb, s):
    return torch.einsum("kj,nja->nka", _rouse(nb), g.reshape(-1, nb, s)).reshape(g.shape)


def _kap64(s, rate=1.0):
    return torch.from_numpy(_shear(s, rate)).to(DEV)


def _grad64(x, h, nb, s, spring):
    _, S = _pairs64(x, h)
    return KBT * S + _force(x, nb, s, spring)


def _implicit64(x, h, nb, s, dt, kap):
    """q+ = q* - (dt/zeta) A g(q+) by its fixed-point iteration."""
    qs = x + dt * _flow(x, nb, s, kap)
    y = qs.clone()
    for _ in range(60):
        z = qs - dt / ZETA * _rouse_mul(_grad64(y, h, nb, s, 0), nb, s)
        done = float((z - y).abs().max()) < 1e-12
        y = z
        if done:
            break
    return y


def _explicit64(x, h, nb, s, spring, dt, kap):
    return x + dt * (_flow(x, nb, s, kap) - _rouse_mul(_grad64(x, h, nb, s, spring), nb, s) / ZETA)


def _median64(x):
    """The lower middle of the N(N-1)/2 distances: a histogram finds the bin, its values are sorted."""
    N = x.shape[0]
    k = (N * (N - 1) // 2 - 1) // 2
    rank = N + 2 * k  # among the N^2 ordered ones, the diagonal first
    top = 4.0 * float((x * x).sum(1).max()) + 1e-9
    bins = 1 << 20 if N > 4000 else 1 << 12
    hist = torch.zeros(bins, dtype=torch.int64, device=DEV)

    def count(sl, r2):
        r2[torch.arange(r2.shape[0], device=DEV), torch.arange(sl.start, sl.stop, device=DEV)] = 0.0
        hist.add_(torch.bincount((r2.reshape(-1) * (bins / top)).long().clamp_(max=bins - 1), minlength=bins))
    _rows64(x, count)
    cum = torch.cumsum(hist, 0)
    b = int((cum <= rank).sum())
    below = int(cum[b - 1]) if b else 0
    vals = []

    def pick(sl, r2):
        r2[torch.arange(r2.shape[0], device=DEV), torch.arange(sl.start, sl.stop, device=DEV)] = 0.0
        f = r2.reshape(-1)
        vals.append(f[(f * (bins / top)).long().clamp_(max=bins - 1) == b])
    _rows64(x, pick)
    return float(torch.sort(torch.cat(vals))[0][rank - below])


def _net64(layers, x):
    for i, (W, b) in enumerate(layers):
        x = x @ W.T + b
        if i < len(layers) - 1:
            x = x * torch.sigmoid(x)
    return x


def _exact_frozen(case, seed):
    N, nb, s, r = case["N"], case["nb"], case["s"], case["r"]
    phi32, P32 = _reduced(case, _gen(seed))
    phi, P, h, dt = phi32.double(), P32.double(), _bandwidth(max(N, 3), nb * s), 0.005
    F = phi.reshape(N, s, r)
    A, kap = _rouse(nb), _kap64(s)
    XH = torch.einsum("nap,ab,nbq->pq", F, kap, F)
    for n in range(case["steps"]):
        if n % case["refresh"] == 0:
            x = torch.einsum("nar,rk->nka", F, P).reshape(N, nb * s)
            rho = torch.empty(N, dtype=torch.float64, device=DEV)

            def first(sl, r2):
                rho[sl] = r2.mul_(-0.5 / (h * h)).exp_().sum(1)
            _rows64(x, first)
            w = 1.0 / rho
            f = F.reshape(N, s * r)
            R = torch.cat([w[:, None], f, w[:, None] * f], 1)
            XB = torch.zeros((r, r), dtype=torch.float64, device=DEV)

            def second(sl, r2):
                V = r2.mul_(-0.5 / (h * h)).exp_() @ R
                U = f[sl] * (1.0 + V[:, :1]) - (w[sl, None] * V[:, 1:s * r + 1] + V[:, s * r + 1:])
                XB.add_(torch.einsum("nap,naq->pq", F[sl], U.reshape(-1, s, r)), alpha=-1.0 / (h * h))
            _rows64(x, second)
        P = P + dt * (XH @ P - KBT / ZETA * XB @ P @ A - P @ A / ZETA)
    return P


def exact(case, seed):
    kind = case["kind"]
    nb, s = case.get("nb", 1), case.get("s", 1)
    if kind == "convect":
        st = prepare(case, seed)
        nx, ny, nz, dt, dx = case["nx"], case["ny"], case["nz"], 0.01, 0.5
        q = st["q"].double().reshape(nz, ny, nx, -1)
        u = st["u"].double().reshape(nz, ny, nx, 3)
        out = q.clone()
        for ax, (dim, n) in enumerate(((2, nx), (1, ny), (0, nz))):
            if n == 1:
                continue
            lo, hi = q.roll(1, dim), q.roll(-1, dim)
            if case["bc"] == 1:
                lo, hi = lo.clone(), hi.clone()
                lo.select(dim, 0).copy_(q.select(dim, 0))
                hi.select(dim, n - 1).copy_(q.select(dim, n - 1))
            v = u[..., ax:ax + 1]
            out -= dt / dx * (v.clamp(min=0.0) * (q - lo) + v.clamp(max=0.0) * (hi - q))
        return out.reshape(st["out"].shape)
    gen = _gen(seed)
    if kind in ("explicit", "implicit"):
        x = _cloud(case["N"], nb, s, case["strain"], gen, case["spring"]).double()
        h = case.get("h") or _bandwidth(case["N"], nb * s)
        for _ in range(case["steps"]):
            if kind == "explicit":
                x = _explicit64(x, h, nb, s, case["spring"], case["dt"], _kap64(s))
            else:
                x = _implicit64(x, h, nb, s, case["dt"], _kap64(s))
        return x
    if kind == "evaluate":
        x = _cloud(case["N"], nb, s, case["strain"], gen, case["spring"]).double()
        N, D = x.shape
        h = _bandwidth(N, D)
        rho, S = _pairs64(x, h)
        n2 = (x.reshape(N, nb, s) ** 2).sum(-1)
        psi = 0.5 * n2 if case["spring"] == 0 else -0.5 * FENE_B * torch.log(1.0 - n2 / FENE_B)
        E = KBT * (torch.log(rho) - math.log(N) - 0.5 * D * math.log(2.0 * math.pi * h * h)) + psi.sum(1)
        return float(E.mean()), KBT * S + _force(x, nb, s, case["spring"]), rho
    if kind == "bandwidth":
        N = case["N"]
        return math.sqrt(_median64(_cloud(N, nb, s, case["strain"], gen).double()) / (2.0 * math.log(N)))
    if kind == "batch":
        sizes, rates = _batch_sizes(case, seed)
        q = _cloud(int(sizes.sum()), nb, s, 0.0, gen).double()
        out, o = [], 0
        for n, rate in zip(sizes, rates):
            x, h = q[o:o + n], _bandwidth(int(n), nb * s)
            for _ in range(case["steps"]):
                if case["scheme"] == 1:
                    x = _implicit64(x, h, nb, s, 0.005, _kap64(s, rate))
                else:
                    x = _explicit64(x, h, nb, s, 0, 0.005, _kap64(s, rate))
            out.append(x)
            o += n
        return torch.cat(out)
    if kind == "pod":
        X = _snapshots(case, gen).double()
        lam, V = torch.linalg.eigh(X @ X.T)
        lam, V = lam.flip(0), V.flip(1)
        r = case["r"]
        phi = X.T @ (V[:, :r] / lam[:r].sqrt())
        at = phi.abs().argmax(0)
        phi = phi * torch.sign(phi[at, torch.arange(r, device=DEV)])
        return dict(r=r, lam=lam.cpu().numpy(), phi=phi)
    if kind == "frozen":
        return _exact_frozen(case, seed)
    if kind == "surrogate":
        N = case["N"]
        phi, P = _reduced(case, gen)
        layers = [(torch.from_numpy(W).double().to(DEV), torch.from_numpy(b).double().to(DEV))
                  for W, b in _score_layers(nb * s, gen)]
        F, P = phi.double().reshape(N, s, case["r"]), P.double()
        for _ in range(case["steps"]):
            x = torch.einsum("nar,rk->nka", F, P).reshape(N, nb * s)
            sc = _net64(layers, x)
            g = KBT * (sc - sc.mean(0)) + x
            v = _flow(x, nb, s, _kap64(s)) - _rouse_mul(g, nb, s) / ZETA
            P = P + 0.005 * torch.einsum("nar,nka->rk", F, v.reshape(N, nb, s))
        return dict(P=P, err=None, fell_back=0)
    # train: denoising score matching and Adam
    x, rows, eps, sigma = _train_draws(case, gen)
    flat = [torch.from_numpy(a).double().to(DEV).requires_grad_(True) for W, b in _train_layers(nb * s, seed)
            for a in (W, b)]
    m, v = [torch.zeros_like(a) for a in flat], [torch.zeros_like(a) for a in flat]
    for k in range(case["steps"]):
        e = eps[k].double()
        r = _net64(list(zip(flat[0::2], flat[1::2])), x[rows[k].long()].double() + sigma * e) + e / sigma
        grads = torch.autograd.grad((r * r).sum(1).mean(), flat)
        with torch.no_grad():
            for a, g, mm, vv in zip(flat, grads, m, v):
                mm.mul_(0.9).add_(g, alpha=0.1)
                vv.mul_(0.999).addcmul_(g, g, value=0.001)
                a -= 1e-3 * (mm / (1 - 0.9 ** (k + 1))) / ((vv / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    flat = [a.detach() for a in flat]
    return list(zip(flat[0::2], flat[1::2]))

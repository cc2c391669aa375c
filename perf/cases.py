"""The calls whose speed this repository is judged by: each case is one pass through the public
binding (paper_1809_10186_gb300.binding), as a program that uses the library makes it.

The workloads are the ones of paper_1809_10186_gb300/workloads.py and bench.py at their own velocity
grids, sphere rules and kernels: the space-homogeneous N = 16 run in FP64, the 1-D slab at N = 24, the
N = 32 batches in every precision that is used in earnest, the differentiation workload, the VSS
kernel and the ragged cavity mesh. Batches run from one node to 2048.

A case is a dict: `kind` (which call), `prec`, `N`, `M` (points of the full-sphere rule), `B` (nodes;
elements for `dg` and `slab`), and `omega`, `alpha`, `svd_tol`, `order`, `steps` where the call has them.
"""
import math

import numpy as np
import torch

from paper_1809_10186_gb300 import binding

PI = math.pi
#: half width of the velocity domain for each grid: the states below are resolved there
HALF_WIDTH = {8: 3.5, 12: 4.0, 16: 5.0, 24: 6.0, 32: 7.0}
K_DG = 3                                          # Gauss-Lobatto nodes of an element (the paper's order 2)
SLAB = dict(L=5.09, Kn=1.582 * 2.0 / PI, T_left=263.0 / 273.0, T_right=283.0 / 273.0, dt=0.002)


def listed():
    return [
        # the smallest call: the collision residual of one node of the space-homogeneous run (FP64, Maxwell
        # molecules, six sphere points), where launches and latency are all there is
        dict(name="collide_f64_n16_b1", kind="collide", prec="fp64", N=16, M=6, B=1, omega=1.0),
        # one SSP-RK3 step of a few dozen nodes on a coarse grid and the moments a solver logs after it
        dict(name="ssprk3_f32_n16_b37", kind="ssprk", prec="fp32", N=16, M=12, B=37, omega=0.81, order=3, steps=1),
        # two SSP-RK2 steps of the 1-D Fourier heat-transfer slab: transport, walls and collisions
        dict(name="slab_f32_n24_i10", kind="slab", prec="fp32", N=24, M=12, B=10, omega=1.0, order=2, steps=2),
        # the collision term of a 1-D mesh of 16 elements x 3 nodes (the slab workload, argon VHS)
        dict(name="dg_f32_n24_e16", kind="dg", prec="fp32", N=24, M=12, B=16, omega=0.81),
        # an FP32 batch on the primary grid
        dict(name="collide_f32_n32_b256", kind="collide", prec="fp32", N=32, M=38, B=256, omega=0.74, svd_tol=1e-8),
        # forward and backward of the differentiation workload: gradients of f and of the VHS exponent
        dict(name="grad_f32_n32_b48", kind="grad", prec="fp32", N=32, M=38, B=48, omega=0.81),
        # the VSS kernel (argon, alpha = 1.40): one transform per radial and sphere point
        dict(name="vss_f32_n32_b40", kind="collide", prec="fp32", N=32, M=38, B=40, omega=0.81, alpha=1.40),
        # the headline batch: 2048 nodes on the tensor cores with 16-bit data
        dict(name="collide_f16s_n32_b2048", kind="collide", prec="f16s", N=32, M=38, B=2048, omega=0.74, svd_tol=1e-8),
        # a batch that lives in pinned host memory, with its copies in and out
        dict(name="host_f16s_n32_b301", kind="host", prec="f16s", N=32, M=38, B=301, omega=0.74, svd_tol=1e-8),
        # the ragged cavity mesh: N = 16, 24, 32 at 40/40/20 % with a VHS exponent for every node
        dict(name="ragged_f16s_b1152", kind="ragged", prec="f16s", N=0, M=26, B=1152),
        # FP32-accurate evaluation on the tensor cores, an odd batch
        dict(name="collide_f16x3_n32_b333", kind="collide", prec="f16x3", N=32, M=38, B=333, omega=0.74, svd_tol=1e-8),
        # a Jacobian-vector product of an implicit or sensitivity solve at the same accuracy
        dict(name="jvp_f16x3_n32_b75", kind="jvp", prec="f16x3", N=32, M=38, B=75, omega=0.81),
    ]


RAGGED_N, RAGGED_SPLIT, RAGGED_OMEGA = (16, 24, 32), (0.4, 0.4, 0.2), (0.5, 0.74, 0.81)


def draw(rng):
    kind = rng.choice(["collide", "collide", "collide", "ssprk", "slab", "dg", "grad", "vss", "host", "ragged", "jvp"])
    logint = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    omega = rng.choice([0.5, 0.74, 0.81, 1.0])
    if kind == "ragged":
        return dict(kind=kind, prec="f16s", N=0, M=rng.choice([12, 26, 38]), B=logint(120, 3000))
    if kind == "slab":
        return dict(kind=kind, prec="fp32", N=rng.choice([16, 24]), M=rng.choice([6, 12]), B=logint(5, 24), omega=omega,
                    order=rng.choice([2, 3]), steps=2)
    if kind == "dg":
        return dict(kind=kind, prec="fp32", N=rng.choice([12, 16, 24, 32]), M=rng.choice([12, 26]), B=logint(8, 40),
                    omega=omega)
    if kind == "vss":
        N = rng.choice([16, 24, 32])
        return dict(kind="collide", prec="fp32", N=N, M=rng.choice([12, 26, 38]), B=logint(16, 8 * 40 * 16 // N), omega=omega,
                    alpha=rng.choice([1.26, 1.40, 1.66]))
    if kind == "grad":
        N = rng.choice([12, 16, 24, 32])
        return dict(kind=kind, prec="fp32", N=N, M=rng.choice([12, 26, 38]), B=logint(16, 64 * 32 // N), omega=omega)
    if kind == "ssprk":
        N = rng.choice([8, 12, 16, 24, 32])
        return dict(kind=kind, prec=rng.choice(["fp32", "fp32", "f16x3"]) if N in (16, 32) else "fp32", N=N,
                    M=rng.choice([6, 12, 26]), B=logint(1, 60), omega=omega, order=rng.choice([2, 3]), steps=rng.choice([1, 2]))
    if kind == "jvp":
        prec = rng.choice(["fp32", "f16x3", "bf16x3"])
        return dict(kind=kind, prec=prec, N=rng.choice([16, 24, 32]), M=rng.choice([12, 26, 38]), B=logint(16, 160), omega=omega)
    prec = "f16s" if kind == "host" else rng.choice(["fp64", "fp32", "fp32", "f16s", "f16x3", "f16x3", "bf16x3"])
    if prec == "fp64":
        N, lo, hi = rng.choice([8, 12, 16]), 1, 48
    elif prec == "fp32":
        N, lo, hi = rng.choice([12, 16, 24, 32]), 16, 500
    else:
        N, lo, hi = rng.choice([16, 24, 32]), 16, (2000 if prec == "f16s" else 700)
    case = dict(kind=kind, prec=prec, N=N, M=rng.choice([6, 12, 26, 38]) if prec in ("fp64", "fp32") else rng.choice([12, 26, 38]),
                B=logint(lo, hi), omega=omega)
    if N == 32:
        case["svd_tol"] = rng.choice([0.0, 1e-8])
    return case


# ---- what a program has in hand before the call --------------------------------------------------

def _grid(N, L, dev="cuda"):
    return -L + (torch.arange(N, dtype=torch.float64, device=dev) + 0.5) * (2.0 * L / N)


def _mixture(B, N, L, seed):
    """(f, M): f [B, N, N, N] FP64, per node a sum of two Maxwellians n (pi T)^-3/2 exp(-|c-u|^2/T) with
    n ~ U[0.5, 1.5], T ~ U[0.7, 1.3], u ~ N(0, 0.5^2): the bimodal states inside a shock or next to a wall;
    M: the Maxwellian of the same density, velocity and temperature."""
    g = torch.Generator().manual_seed(int(seed))
    n = (0.5 + torch.rand(B, 2, 1, generator=g, dtype=torch.float64)).cuda()
    u = (0.5 * torch.randn(B, 2, 3, generator=g, dtype=torch.float64)).cuda()
    T = (0.7 + 0.6 * torch.rand(B, 2, 1, generator=g, dtype=torch.float64)).cuda()

    def field(n, u, T):
        e = torch.exp(-((_grid(N, L) - u[..., None]) ** 2) / T[..., None])        # [B, s, 3, N]
        e[:, :, 0] *= n / (PI * T) ** 1.5
        return torch.einsum("bsx,bsy,bsz->bxyz", e[:, :, 0], e[:, :, 1], e[:, :, 2])
    n0 = n.sum(1, keepdim=True)
    u0 = (n * u).sum(1, keepdim=True) / n0
    T0 = (n * (T + 2.0 / 3.0 * ((u - u0) ** 2).sum(2, keepdim=True))).sum(1, keepdim=True) / n0
    return field(n, u, T), field(n0, u0, T0)


def _unit(d):
    return d / d.flatten(1).norm(dim=1).reshape(-1, 1, 1, 1)


def _bkw(N, L, t):
    c = _grid(N, L)
    c2 = c[:, None, None] ** 2 + c[None, :, None] ** 2 + c[None, None, :] ** 2
    K = 1.0 - math.exp(-t / 6.0)
    return (torch.exp(-c2 / (2 * K)) / (2 * (2 * PI * K) ** 1.5) * ((5 * K - 3) / K + (1 - K) / K ** 2 * c2))[None]


def _inputs(case, seed):
    """The fields of a case in FP64, already rounded to the type that the plan takes."""
    kind, N, B = case["kind"], case["N"], case["B"]
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    rounded = lambda x: x.to(dt)
    if kind == "ragged":
        g = np.random.Generator(np.random.Philox(int(seed)))
        counts = [int(round(B * s)) for s in RAGGED_SPLIT]
        counts[-1] = B - sum(counts[:-1])
        node_N = np.concatenate([np.full(c, n) for c, n in zip(counts, RAGGED_N)])[g.permutation(B)]
        node_omega = np.asarray(RAGGED_OMEGA)[g.integers(0, 3, size=B)]
        offset = np.concatenate([[0], np.cumsum(node_N.astype(np.int64) ** 3)])
        f = torch.empty(int(offset[-1]), dtype=dt, device="cuda")
        for k, n in enumerate(RAGGED_N):
            idx = np.nonzero(node_N == n)[0]
            at = torch.from_numpy(offset[idx]).cuda()[:, None] + torch.arange(n ** 3, device="cuda")
            f[at.reshape(-1)] = rounded(_mixture(len(idx), n, HALF_WIDTH[n], seed + 101 * k)[0]).reshape(-1)
        return dict(f=f, node_N=node_N, node_omega=node_omega, offset=offset[:-1])
    if kind == "slab":
        # a state near the initial Maxwellian n = 1, T = 1 of the slab, varying from node to node
        g = torch.Generator().manual_seed(int(seed))
        x = _grid(N, SLAB["L"])
        r = lambda: torch.rand(B * K_DG, 1, generator=g, dtype=torch.float64).cuda()
        n, T, ux = 0.9 + 0.2 * r(), 0.95 + 0.1 * r(), 0.1 * (r() - 0.5)
        e = torch.exp(-x ** 2 / T)
        f = torch.einsum("bx,by,bz->bxyz", torch.exp(-(x - ux) ** 2 / T) * n / (PI * T) ** 1.5, e, e)
        return dict(f=rounded(f).reshape(B, K_DG, N, N, N))
    L = HALF_WIDTH[N]
    if kind == "collide" and case["prec"] == "fp64" and case["M"] == 6 and B == 1:
        return dict(f=rounded(_bkw(N, _half_width(case), 5.5 + (seed % 997) / 997.0)))
    f, equilibrium = _mixture(B * K_DG if kind == "dg" else B, N, L, seed)
    if kind == "dg":
        return dict(f=rounded(f).reshape(B, K_DG, N, N, N))
    out = dict(f=rounded(f))
    if kind == "grad":      # the cotangent of a misfit of relaxation rates: along M - f, as Q itself
        out["v"] = rounded(_unit(equilibrium - f))
    elif kind == "jvp":     # a tangent: the difference of two states
        out["v"] = rounded(_unit(_mixture(B, N, L, seed + 7919)[0] - f))
    return out


def _half_width(case):
    if case["kind"] == "slab":
        return SLAB["L"]
    if case["prec"] == "fp64" and case["M"] == 6 and case["B"] == 1 and case["N"] == 16:
        return 8.0                                # the BKW workload's own domain
    return HALF_WIDTH[case["N"]]


def _gamma(omega):
    return 2.0 * (1.0 - omega)


def _plan(case, N, L, omega):
    nodes = case["B"] if case["kind"] not in ("slab", "dg", "ragged") else 0
    return binding.Plan(N=N, L=L, gamma=_gamma(omega), M=case["M"], N_rho=N, svd_tol=case.get("svd_tol", 0.0),
                        precision=case["prec"], alpha=case.get("alpha", 0.0), max_batch=nodes if nodes > 1024 else 0)


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, N, B = case["kind"], case["N"], case["B"]
    if kind == "ragged":
        plans = [_plan(case, n, HALF_WIDTH[n], 0.74) for n in RAGGED_N]
        node_plan = np.searchsorted(np.asarray(RAGGED_N), x["node_N"]).astype(np.int32)
        gam = _gamma(x["node_omega"])
        b = np.asarray([_kernel_constant(w) for w in x["node_omega"]])
        return dict(kind=kind, f=x["f"], call=binding.RaggedSchedule(plans, node_plan, x["offset"], gam, b))
    plan = _plan(case, N, _half_width(case), case["omega"])
    st = dict(kind=kind, plan=plan, f=x["f"], v=x.get("v"))
    if kind == "dg":
        st["call"] = binding.DGElement(plan, binding.host_dg_tensor(K_DG)[2], max_elements=B)
    elif kind == "slab":
        st["call"] = binding.Slab(plan, K_DG, np.linspace(0.0, 1.0, B + 1), SLAB["Kn"], (0, 0, 0, SLAB["T_left"]),
                                  (0, 0, 0, SLAB["T_right"]))
        st["order"], st["steps"] = case["order"], case["steps"]
    elif kind == "ssprk":
        st["order"], st["steps"] = case["order"], case["steps"]
    elif kind == "grad":
        st["f"].requires_grad_(True)
        st["gamma"] = torch.full((B,), _gamma(case["omega"]), dtype=torch.float64, device="cuda", requires_grad=True)
    elif kind == "host":
        st["f"] = x["f"].cpu().pin_memory()
        st["q"] = torch.empty_like(st["f"]).pin_memory()
    return st


def run(state):
    kind, plan = state["kind"], state.get("plan")
    if kind == "collide":
        return plan.collide(state["f"])
    if kind == "host":
        return plan.collide_host(state["f"], state["q"])
    if kind in ("ragged", "dg"):
        return state["call"].collide(state["f"])
    if kind == "slab":
        return state["call"].ssprk(state["f"], SLAB["dt"], state["steps"], order=state["order"])
    if kind == "ssprk":
        f = plan.ssprk(state["f"], 0.02, state["steps"], order=state["order"])
        return f, plan.moments(f)
    if kind == "jvp":
        return plan.collide_jvp(state["f"], state["v"])
    Q = binding.collide(plan, state["f"], state["gamma"])
    gf, gg = torch.autograd.grad(Q, (state["f"], state["gamma"]), state["v"])
    return Q.detach(), gf, gg


def work(case):
    """Bytes: every input field read once, every output written once. Flops: the method's own count, one
    complex transform of N^3 points (5 N^3 log2 N^3) and 20 N^3 for phases and products per radial point and
    sphere pair and evaluation (7.5 N^3 log2 N^3 + 20 N^3 where the kernel keeps the sphere point; twice the
    transforms for a tangent or adjoint, whose operands are two fields)."""
    kind, B, M, es = case["kind"], case["B"], case["M"], 8 if case["prec"] == "fp64" else 4
    per = lambda n, c: n * (M // 2) * (c * n ** 3 * math.log2(n ** 3) + 20.0 * n ** 3)
    if kind == "ragged":
        counts = [B * s for s in RAGGED_SPLIT]
        return dict(bytes=sum(2 * es * c * n ** 3 for c, n in zip(counts, RAGGED_N)),
                    flops=sum(c * per(n, 5.0) for c, n in zip(counts, RAGGED_N)))
    N = case["N"]
    n3 = N ** 3
    one = per(N, 7.5 if case.get("alpha", 0.0) not in (0.0, 1.0) else 5.0)
    stages = case.get("order", 1) * case.get("steps", 1)
    if kind == "dg":
        return dict(bytes=2 * es * B * K_DG * n3, flops=B * K_DG * K_DG * one)
    if kind == "slab":
        return dict(bytes=2 * es * B * K_DG * n3, flops=stages * B * K_DG * K_DG * one)
    if kind == "ssprk":
        return dict(bytes=2 * es * B * n3 + 120 * B, flops=stages * B * one)
    if kind == "grad":
        return dict(bytes=4 * es * B * n3 + 16 * B, flops=B * (one + per(N, 10.0)))
    if kind == "jvp":
        return dict(bytes=3 * es * B * n3, flops=B * per(N, 10.0))
    return dict(bytes=2 * es * B * n3, flops=B * one)


# ---- the same results in 64 bits, with torch alone ----------------------------------------------

def _kernel_constant(omega, alpha=1.0):
    """b of the VHS (alpha = 1) or VSS kernel."""
    return alpha / (2.0 ** (2.0 - omega + alpha) * math.gamma(2.5 - omega) * PI)


def _sphere(M):
    """(points [P, 3], weights [P]) of one point for each antipodal pair of the M-point rule."""
    def orbit(*v):
        import itertools
        pts = {tuple(s * c + 0.0 for s, c in zip(sg, p)) for p in itertools.permutations(v) for sg in itertools.product((1, -1), repeat=3)}
        return sorted({tuple(0.0 if c == 0 else c for c in p) for p in pts})
    if M == 12:
        phi = 0.5 * (1 + math.sqrt(5.0))
        n = math.sqrt(1 + phi * phi)
        base = [(0.0, s / n, t * phi / n) for s in (1, -1) for t in (1, -1)]
        sets = [(p, 4 * PI / 12) for q in base for p in (q, (q[1], q[2], q[0]), (q[2], q[0], q[1]))]
    else:
        s2, s3 = math.sqrt(0.5), math.sqrt(1 / 3.0)
        # weights as fractions of the sphere: octahedron, 26-point and 38-point Lebedev rules
        q = 0.4597008433809831
        rules = {6: [((1.0, 0.0, 0.0), 1 / 6)],
                 26: [((1.0, 0.0, 0.0), 1 / 21), ((s2, s2, 0.0), 4 / 105), ((s3, s3, s3), 9 / 280)],
                 38: [((1.0, 0.0, 0.0), 1 / 105), ((s3, s3, s3), 9 / 280), ((q, math.sqrt(1 - q * q), 0.0), 1 / 35)]}
        sets = [(p, 4 * PI * w) for v, w in rules[M] for p in orbit(*v)]
    first = lambda p: next(c for c in p if abs(c) > 1e-14) > 0
    sets = [(p, w) for p, w in sets if first(p)]
    return np.asarray([p for p, _ in sets]), np.asarray([w for _, w in sets])


def _sph_bessel(top, a):
    """j_0 .. j_top of a [n] (a >= 0): downward recurrence, normalised with sum (2l+1) j_l^2 = 1."""
    a0, a = a, a.clamp(min=1e-4)
    start = int(max(float(a.max()), top)) + 90
    out = torch.zeros(top + 1, *a.shape, dtype=torch.float64, device=a.device)
    hi, cur = torch.zeros_like(a), torch.full_like(a, 1e-100)
    norm = (2 * start + 1) * cur ** 2
    for l in range(start, 0, -1):
        if l <= top:
            out[l] = cur
        hi, cur = cur, (2 * l + 1) / a * cur - hi
        big = cur.abs() > 1e60
        s = torch.where(big, torch.full_like(a, 1e-60), torch.ones_like(a))
        hi, cur, norm, out = hi * s, cur * s, norm * s * s, out * s
        norm = norm + (2 * l - 1) * cur ** 2
    out[0] = cur
    out = out / norm.sqrt()
    j0, j1 = torch.sin(a) / a, torch.sin(a) / a ** 2 - torch.cos(a) / a
    flip = torch.where(j0.abs() >= j1.abs(), j0 * out[0], j1 * out[1]) < 0
    out = torch.where(flip, -out, out)
    out[:, a0 < 1e-4] = 0.0
    out[0, a0 < 1e-4] = 1.0
    return out


class _Operator:
    """The fast spectral collision operator in FP64, by torch.fft."""

    def __init__(self, N, L, M, omega, alpha=0.0):
        self.N, self.L, self.gamma = N, L, _gamma(omega)
        self.vss = alpha not in (0.0, 1.0)
        self.alpha, self.b = (alpha, _kernel_constant(omega, alpha)) if self.vss else (1.0, _kernel_constant(omega))
        R = 4.0 * L / (3.0 + math.sqrt(2.0))
        x, w = np.polynomial.legendre.leggauss(N)
        self.cr, self.wr = 0.5 * R * (x + 1.0), 0.5 * R * w
        self.sigma, self.wsig = _sphere(M)
        k = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device="cuda")
        self.k = k
        self.kabs = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2).sqrt()
        self.rho = 4 * PI * self.b * self.cr ** (self.gamma + 2.0)
        self.radial = lambda r, f=1.0: f * self.wr[r] * self.rho[r] * torch.sinc(self.cr[r] * self.kabs / (2 * L))
        if self.vss:
            self.factors = [self._vss_factors(r) for r in range(N)]
            self.loss = sum(g for _, g in self.factors)
        else:
            self.loss = self._loss(np.ones(N))

    def _loss(self, f):
        return sum(4 * PI * f[r] * self.wr[r] * self.rho[r] * torch.sinc(self.cr[r] * self.kabs / self.L) for r in range(self.N))

    def _vss_factors(self, r):
        """w_r w_p F(k, c_r, sigma_p) for every p, and the loss weight's share of r."""
        beta, pref = self.alpha - 1.0, 2 * PI * self.b * self.cr[r] ** (self.gamma + 2.0)
        kv = torch.stack(torch.meshgrid(self.k, self.k, self.k, indexing="ij"), -1)
        sig = torch.from_numpy(self.sigma).cuda()
        mu = torch.where(self.kabs[..., None] > 0, (kv @ sig.T) / self.kabs[..., None].clamp(min=1.0), 0.0).movedim(-1, 0)
        q2, inv = torch.unique((self.kabs ** 2).round().long(), return_inverse=True)
        q = q2.double().sqrt()
        out = []
        for arg in (PI * self.cr[r] * q / (2 * self.L), PI * self.cr[r] * q / self.L):
            top = 2 * ((int(float(arg.max())) + 44) // 2)
            j = _sph_bessel(top, arg)
            c, acc, pm, pc = 2.0 ** (beta + 1) / (beta + 1), 0.0, torch.ones_like(mu), mu
            for l in range(top + 1):
                P = pm if l == 0 else pc
                if l % 2 == 0:
                    acc = acc + ((2 * l + 1) * c * (-1) ** (l // 2) * j[l])[inv] * P
                c *= (beta - l) / (beta + l + 2.0)
                if l >= 1:
                    pm, pc = pc, ((2 * l + 1) * mu * pc - l * pm) / (l + 1)
            out.append(pref * self.wr[r] * acc)
        w = torch.from_numpy(self.wsig).cuda()[:, None, None, None]
        return w * out[0], (2 * w * out[1]).sum(0)

    def _phase(self, r, p):
        m = []
        for s in 0.5 * self.cr[r] * self.sigma[p]:
            e = torch.polar(torch.ones_like(self.k), PI * self.k * float(s) / self.L)
            e[self.N // 2] = math.cos(PI * self.N * float(s) / (2 * self.L))
            m.append(e)
        return m[0][:, None, None] * m[1][None, :, None] * m[2][None, None, :]

    def _gain(self, f, g, scale):
        """Spectrum of sum_r K_r sum_p w_p [(T_s f)(T_-s g) + (T_-s f)(T_s g)]."""
        F = torch.fft.fftn(f, dim=(1, 2, 3))
        G = F if g is f else torch.fft.fftn(g, dim=(1, 2, 3))
        total = torch.zeros_like(F)
        for r in range(self.N):
            P = torch.zeros_like(f)
            for p in range(len(self.wsig)):
                m = self._phase(r, p)
                if g is f:
                    z = torch.fft.ifftn(F * (m + 1j * m.conj()), dim=(1, 2, 3))
                    pr = 2 * z.real * z.imag
                else:
                    z = torch.fft.ifftn(F * m + 1j * (G * m.conj()), dim=(1, 2, 3))
                    y = torch.fft.ifftn(F * m.conj() + 1j * (G * m), dim=(1, 2, 3))
                    pr = z.real * z.imag + y.real * y.imag
                if self.vss:
                    total += self.factors[r][0][p] * torch.fft.fftn(pr, dim=(1, 2, 3))
                else:
                    P += self.wsig[p] * pr
            if not self.vss:
                total += self.radial(r, scale[r]) * torch.fft.fftn(P, dim=(1, 2, 3))
        return total

    def _conv(self, W, x):
        return torch.fft.ifftn(W * torch.fft.fftn(x, dim=(1, 2, 3)), dim=(1, 2, 3)).real

    def _chunks(self, fn, *fields):
        c = max(1, 3 * 10 ** 9 // (16 * self.N ** 3 * 8))
        return torch.cat([fn(*(x[i:i + c] for x in fields)) for i in range(0, fields[0].shape[0], c)])

    def collide(self, f, g=None, scale=None):
        one = np.ones(self.N) if scale is None else scale
        loss = self.loss if scale is None else self._loss(scale)

        def part(f, g):
            return torch.fft.ifftn(self._gain(f, g, one), dim=(1, 2, 3)).real - f * self._conv(loss, g)
        return self._chunks(lambda f: part(f, f), f) if g is None else self._chunks(part, f, g)

    def jvp(self, f, v):
        return self.collide(f, v) + self.collide(v, f)

    def dgamma(self, f):
        return self.collide(f, scale=np.log(self.cr))

    def vjp(self, f, u):
        def part(f, u):
            F, out = torch.fft.fftn(f, dim=(1, 2, 3)), 0.0
            back = torch.zeros_like(F)
            for r in range(self.N):
                ur = self._conv(self.radial(r), u)
                for p in range(len(self.wsig)):
                    m = self._phase(r, p)
                    z = torch.fft.ifftn(F * (m + 1j * m.conj()), dim=(1, 2, 3))
                    # T_-s(u_r T_-s f) + T_s(u_r T_s f), s = +: real part, s = -: imaginary part
                    back += 2 * self.wsig[p] * (m.conj() * torch.fft.fftn(ur * z.imag, dim=(1, 2, 3)) +
                                                m * torch.fft.fftn(ur * z.real, dim=(1, 2, 3)))
            out = torch.fft.ifftn(back, dim=(1, 2, 3)).real
            return out - u * self._conv(self.loss, f) - self._conv(self.loss, u * f)
        return self._chunks(part, f, u)


def _stepped(rhs, f, dt, order, steps):
    for _ in range(steps):
        a = f + dt * rhs(f)
        if order == 2:
            f = 0.5 * f + 0.5 * a + 0.5 * dt * rhs(a)
        else:
            a = 0.75 * f + 0.25 * a + 0.25 * dt * rhs(a)
            f = f / 3.0 + 2.0 / 3.0 * a + 2.0 / 3.0 * dt * rhs(a)
    return f


def _moments(f, N, L):
    """n, u, T, P_xx .. P_yz, q, H of every node by the mid-point rule."""
    c = _grid(N, L)
    dv = (2.0 * L / N) ** 3
    C = torch.stack(torch.meshgrid(c, c, c, indexing="ij"))
    n = f.sum((1, 2, 3)) * dv
    u = torch.einsum("axyz,bxyz->ba", C, f) * dv / n[:, None]
    d = C[None] - u[:, :, None, None, None]
    d2 = (d * d).sum(1)
    T = 2.0 / (3.0 * n) * (f * d2).sum((1, 2, 3)) * dv
    P = [2.0 * (d[:, i] * d[:, j] * f).sum((1, 2, 3)) * dv for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    q = [(d[:, i] * d2 * f).sum((1, 2, 3)) * dv for i in range(3)]
    H = torch.where(f > 0, f * torch.log(torch.where(f > 0, f, 1.0)), 0.0).sum((1, 2, 3)) * dv
    return torch.stack([n, u[:, 0], u[:, 1], u[:, 2], T, *P, *q, H], 1)


def _dg_basis():
    """M, S, H of the three-node Gauss-Lobatto basis on [-1, 1] (nodes -1, 0, 1), by quadrature."""
    x, w = np.polynomial.legendre.leggauss(6)
    phi = np.stack([x * (x - 1) / 2, 1 - x * x, x * (x + 1) / 2])
    dphi = np.stack([x - 0.5, -2 * x, x + 0.5])
    return (np.einsum("aq,bq,q->ab", phi, phi, w), np.einsum("lq,mq,q->ml", phi, dphi, w),
            np.einsum("aq,bq,cq,q->abc", phi, phi, phi, w))


def _element_term(op, F):
    """C[e, m] = sum H[m, a, b] Q(F[e, a], F[e, b]); every H[m] is symmetric: a sum of quadratic terms."""
    E, K, N = F.shape[0], F.shape[1], F.shape[2]
    H = _dg_basis()[2]
    C = []
    for m in range(K):
        lam, V = np.linalg.eigh(H[m])
        comb = torch.einsum("ar,eaxyz->rexyz", torch.from_numpy(V).to(F), F).reshape(K * E, N, N, N)
        Q = op.collide(comb).reshape(K, E, N, N, N)
        C.append(torch.einsum("r,rexyz->exyz", torch.from_numpy(lam).to(F), Q))
    return torch.stack(C, 1)


def _slab_rhs(op, F):
    I, K, N = F.shape[0], F.shape[1], F.shape[2]
    Mm, S, _ = (torch.from_numpy(a).to(F) for a in _dg_basis())
    x = _grid(N, SLAB["L"])
    c1 = x[:, None, None].expand(N, N, N)
    c2 = x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2
    wall = []
    for T, f, cn in ((SLAB["T_left"], F[0, 0], -c1), (SLAB["T_right"], F[-1, -1], c1)):
        fw = torch.exp(-c2 / T)
        wall.append(-(cn * f)[cn >= 0].sum() / (cn * fw)[cn < 0].sum() * fw)
    left = torch.cat([wall[0][None], F[:-1, -1]])
    right = torch.cat([F[1:, 0], wall[1][None]])
    out = c1 * torch.einsum("ml,ilxyz->imxyz", S, F)
    out[:, -1] -= c1 * torch.where(c1 >= 0, F[:, -1], right)
    out[:, 0] += c1 * torch.where(-c1 >= 0, F[:, 0], left)
    return torch.einsum("ml,ilxyz->imxyz", torch.linalg.inv(Mm), 2.0 * I * out + _element_term(op, F) / SLAB["Kn"])


def exact(case, seed):
    x = _inputs(case, seed)
    kind, N, M = case["kind"], case["N"], case["M"]
    f = x["f"].double()
    if kind == "ragged":
        out = torch.empty_like(f)
        for n in RAGGED_N:
            for w in RAGGED_OMEGA:
                idx = np.nonzero((x["node_N"] == n) & (x["node_omega"] == w))[0]
                if len(idx):
                    at = (torch.from_numpy(x["offset"][idx]).cuda()[:, None] + torch.arange(n ** 3, device="cuda")).reshape(-1)
                    out[at] = _Operator(n, HALF_WIDTH[n], M, w).collide(f[at].reshape(-1, n, n, n)).reshape(-1)
        return out
    L = _half_width(case)
    op = _Operator(N, L, M, case["omega"], case.get("alpha", 0.0))
    if kind in ("collide", "host"):
        q = op.collide(f)
        return q.cpu() if kind == "host" else q
    if kind == "dg":
        return _element_term(op, f)
    if kind == "slab":
        return _stepped(lambda F: _slab_rhs(op, F), f, SLAB["dt"], case["order"], case["steps"])
    if kind == "ssprk":
        f = _stepped(op.collide, f, 0.02, case["order"], case["steps"])
        return f, _moments(f, N, L)
    v = x["v"].double()
    if kind == "jvp":
        return op.jvp(f, v)
    return op.collide(f), op.vjp(f, v), (v * op.dgamma(f)).sum((1, 2, 3))

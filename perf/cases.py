"""Performance cases: the calls a user of this solver makes, through its Python
binding, over the range of its workloads.

Four kinds of pass, each on one of the four flows of the repository (the 2D
isentropic vortex, the 2D viscous cylinder, the inviscid sphere shell and the
viscous extruded ellipse on hexahedra):

* ``residual``  one evaluation of the spatial residual for a state in device
  memory: what an explicit or matrix-free program calls in its inner loop;
* ``cycles``    ten pseudo-iterations of an implicit stage, the first of which
  rebuilds the smoother (``refresh_every = 10``, the default);
* ``step``      one whole ESDIRK3 step, every stage to a 1e-8 drop;
* ``blocks``    a program's own element blocks: upload, factor, apply.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1908_03972_gb300 import pmgfr, workloads as W

PREC = {"fp64": pmgfr.PMG_PREC_FP64, "fp32": pmgfr.PMG_PREC_FP32, "bf16": pmgfr.PMG_PREC_BF16R}
OMEGA = 1767732205903.0 / 4055673282236.0   # diagonal coefficient of ESDIRK3
GAMMA, PR = 1.4, 0.72
SMOOTH = (5, 10, 20, 40)                    # sweeps per level, finest first


def listed():
    return [
        # an explicit program's right-hand side on the small vortex: launches and latency only
        dict(name="residual vortex 8x8 P2", kind="residual", flow="vortex", a=8, b=8, c=0, levels="2", curved=False),
        # the same on a ragged curved mesh at high order
        dict(name="residual vortex 37x29 P5 curved", kind="residual", flow="vortex", a=37, b=29, c=0, levels="5",
             curved=True),
        # the full-size cylinder at P = 4: viscous terms and boundary faces
        dict(name="residual cylinder 64x256 P4", kind="residual", flow="cylinder", a=64, b=256, c=0, levels="4"),
        # viscous hexahedra at P = 3, the matrix-free product of the Newton-Krylov solver
        dict(name="residual ellipse 16x24x8 P3", kind="residual", flow="ellipse", a=16, b=24, c=8, levels="3"),
        # the headline workload's pseudo-iterations in the default mixed arithmetic
        dict(name="cycles vortex 64x64 P3210 fp32", kind="cycles", flow="vortex", a=64, b=64, c=0, levels="3-2-1-0",
             blocks="fp32", flux="dw", curved=False),
        # the same in plain binary64, the arithmetic the mixed one is compared with
        dict(name="cycles vortex 64x64 P3210 fp64", kind="cycles", flow="vortex", a=64, b=64, c=0, levels="3-2-1-0",
             blocks="fp64", flux="fp64", curved=False),
        # the full-size cylinder, P{4-2-1}, BF16 blocks
        dict(name="cycles cylinder 64x256 P421 bf16", kind="cycles", flow="cylinder", a=64, b=256, c=0,
             levels="4-2-1", blocks="bf16", flux="dw"),
        # the sphere shell at 1/16 of its full size, P{2-1-0}
        dict(name="cycles sphere 6x4x4x24 P210 fp32", kind="cycles", flow="sphere", a=4, b=24, c=0, levels="2-1-0",
             blocks="fp32", flux="fp64"),
        # the extruded ellipse, P{3-2-1-0}: blocks of 320 unknowns
        dict(name="cycles ellipse 12x16x5 P3210 fp32", kind="cycles", flow="ellipse", a=12, b=16, c=5,
             levels="3-2-1-0", blocks="fp32", flux="fp64"),
        # one whole step of the small vortex by pseudo-transient continuation
        dict(name="step vortex 8x8 P210 ptc", kind="step", flow="vortex", a=8, b=8, c=0, levels="2-1-0",
             blocks="fp32", flux="dw", solver="ptc", curved=False),
        # one whole step of the headline workload by Newton-Krylov
        dict(name="step vortex 64x64 P3210 nk", kind="step", flow="vortex", a=64, b=64, c=0, levels="3-2-1-0",
             blocks="fp32", flux="dw", solver="nk", curved=False),
        # blocks of a program's own (135 unknowns: hexahedra at P = 2) factored and applied in binary64
        dict(name="blocks hex 768 P2 fp64", kind="blocks", flow="box3", a=12, b=8, c=8, levels="2", blocks="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("residual", "cycles", "cycles", "step", "blocks"))
    if kind == "blocks":
        P = rng.choice((1, 2, 2, 3))
        most = {1: 12, 2: 9, 3: 6}[P]
        return dict(kind=kind, flow="box3", a=_log(rng, 2, most), b=_log(rng, 2, most), c=_log(rng, 2, most),
                    levels=str(P), blocks=rng.choice(("fp64", "fp32")))
    if kind == "step":
        solver = rng.choice(("ptc", "nk"))
        most = 7 if solver == "ptc" else 56
        a = _log(rng, 4, most)
        b = min(most, max(4, int(a * rng.uniform(0.6, 1.5))))   # elements of moderate aspect ratio
        return dict(kind=kind, flow="vortex", a=a, b=b, c=0,
                    levels=rng.choice(("2-1-0", "3-2-1-0") if solver == "nk" else ("2-1-0",)),
                    blocks=rng.choice(("fp32", "bf16") if solver == "ptc" else ("fp32", "fp32", "fp64")), flux="dw",
                    solver=solver, curved=False)
    flow = rng.choice(("vortex", "vortex", "cylinder", "sphere", "ellipse"))
    a, b, c = {"vortex": (_log(rng, 5, 64), _log(rng, 5, 64), 0),
               "cylinder": (_log(rng, 8, 48), _log(rng, 24, 192), 0),
               "sphere": (_log(rng, 2, 4), _log(rng, 5, 24), 0),
               "ellipse": (_log(rng, 5, 12), _log(rng, 8, 16), _log(rng, 2, 5))}[flow]
    case = dict(kind=kind, flow=flow, a=a, b=b, c=c)
    if flow == "vortex":
        case["curved"] = rng.random() < 0.5
    if kind == "residual":
        # hexahedra stop at P = 3; curved meshes need P >= 2 with the gauge pressure
        return dict(case, levels=str({"vortex": rng.randint(2, 5), "cylinder": rng.randint(2, 4),
                                      "sphere": rng.randint(2, 3), "ellipse": rng.randint(2, 3)}[flow]))
    levels = {"vortex": rng.choice(("2-1-0", "3-2-1-0", "4-2-1")), "cylinder": rng.choice(("4-2-1", "3-2-1", "2-1")),
              "sphere": rng.choice(("2-1-0", "2-1")), "ellipse": rng.choice(("3-2-1-0", "2-1-0", "3-1"))}[flow]
    return dict(case, levels=levels, blocks=rng.choice(("fp32", "fp32", "bf16", "fp64")),
                flux=rng.choice(("dw", "dw", "fp64")) if flow == "vortex" else "dw")


# ------------------------------------------------------------------ workloads
@functools.lru_cache(maxsize=32)
def _mesh(flow, a, b, c, curved):
    if flow == "vortex":
        return W.periodic_box(a, b, Ng=2, perturb=0.3) if curved else W.periodic_box(a, b, Ng=1)
    if flow == "cylinder":
        return W.cylinder_omesh(a, b, 0.5, 50.0, Ng=2)
    if flow == "sphere":
        return W.cubed_sphere_shell(a, b, 0.5, 20.0, Ng=2)
    if flow == "ellipse":
        return W.extruded_ellipse(a, b, c, span=0.2, Ng=2)
    return W.periodic_box3d(a, b, c, Ng=1)


def _setup(case):
    """Mesh, dimension, levels and the solver's settings of a case."""
    flow = case["flow"]
    nodes, nbr = _mesh(flow, case["a"], case["b"], case["c"], bool(case.get("curved")))
    levels = [int(p) for p in case["levels"].split("-")]
    if flow in ("vortex", "box3"):
        T, kw = W.freestream_T(0.005), dict(Ma_inf=0.005)
        kw["res_scale" if flow == "vortex" else "res_scale3"] = (
            W.freestream_scales if flow == "vortex" else W.freestream_scales3)(0.005)
        inf = None
    elif flow == "cylinder":
        T = W.freestream_T(0.001, speed=1.0)
        inf = (T, 1.0, 0.0, T)
        kw = dict(Ma_inf=0.001, mu=0.01, cutoff=1, kappa=1.0, q_inf=inf,
                  res_scale=W.freestream_scales(0.001, speed=1.0))
    else:
        Ma = 0.001 if flow == "sphere" else 0.1
        T, al = W.freestream_T(Ma, speed=1.0), math.radians(0.0 if flow == "sphere" else 8.0)
        inf = (T, math.cos(al), math.sin(al), 0.0, T)
        kw = dict(Ma_inf=Ma, cutoff=1, kappa=1.0, q_inf3=inf, res_scale3=W.freestream_scales3(Ma, speed=1.0))
        if flow == "ellipse":
            kw["mu"] = 1.0 / 60000.0
    dim = 2 if flow in ("vortex", "cylinder") else 3
    return nodes, nbr, dim, levels, T, inf, dict(kw, dim=dim, p_gauge=T)


def _state(case, xyz, T, inf, seed):
    """The flow's start with a seeded part: the vortex's place, the noise or the waves of the perturbation."""
    rng = np.random.default_rng(seed)
    flow = case["flow"]
    E, N = xyz.shape[:2]
    if flow == "vortex":
        q = W.isentropic_vortex(xyz, center=tuple(rng.uniform(2.0, 8.0, 2)))
        if case["kind"] == "residual":   # an iterate or a matrix-free product's argument, not a smooth solution
            q[:3] += 0.05 * rng.standard_normal((3, E, N))
            q[3] += 5e-5 * rng.standard_normal((E, N))
        return q
    if flow == "cylinder":
        q = W.freestream_noise_state(xyz, 0.001, seed=seed)
        q[1] *= 1.0 - np.exp(-(np.hypot(xyz[..., 0], xyz[..., 1]) - 0.5) * 4.0)   # a boundary layer
        return q
    q = W.uniform_state3(E, N, T, inf[1], inf[2], inf[3], T)
    if flow == "ellipse":
        q[2] += 1e-3 * rng.standard_normal((E, N))
    else:
        for v in range(3):
            q[1 + v] += 1e-2 * np.sin(xyz @ rng.uniform(0.2, 0.6, 3))
        q[0] *= 1 + 1e-7 * np.cos(xyz[..., 0])
        q[4] *= 1 + 1e-7 * np.sin(xyz[..., 1])
    return q


def _cons(q):
    """Conservative variables of a primitive device state."""
    rho = q[0] / q[-1]
    return torch.stack([rho] + [rho * u for u in q[1:-1]] +
                       [rho * (q[-1] / (GAMMA - 1.0) + 0.5 * (q[1:-1] ** 2).sum(0))])


def _own_blocks(case, seed):
    """Blocks and right-hand sides of the blocks cases: well-conditioned
    matrices whose rows and columns carry the scales of low-Mach equations."""
    E = case["a"] * case["b"] * case["c"]
    N = (int(case["levels"]) + 1) ** 3
    n = 5 * N
    g = torch.Generator(device="cuda").manual_seed(seed)
    D = torch.randn(E, n, n, generator=g, device="cuda", dtype=torch.float64) / math.sqrt(n)
    D.diagonal(dim1=1, dim2=2).add_(2.0)
    scale = torch.tensor([1.0, 1.0, 1.0, 1.0, 3e4], device="cuda", dtype=torch.float64).repeat_interleave(N)
    D *= scale[None, :, None] / scale[None, None, :].flip(2)
    r = torch.randn(5, E, N, generator=g, device="cuda", dtype=torch.float64)
    r[4] *= 3e4
    return D, r


def prepare(case, seed):
    pmgfr.load()
    nodes, nbr, dim, levels, T, inf, kw = _setup(case)
    kind = case["kind"]
    if kind in ("cycles", "step"):
        kw["flux_prec"] = pmgfr.PMG_FLUX_FP64 if case["flux"] == "fp64" else pmgfr.PMG_FLUX_DW_SMOOTH
    if "blocks" in case:
        kw["block_prec"] = PREC[case["blocks"]]
    s = pmgfr.Solver(nodes, nbr, levels, list(SMOOTH[:len(levels)]), tol=1e-8, **kw)
    st = dict(kind=kind, s=s)
    if kind == "blocks":
        st["D"], st["r"] = _own_blocks(case, seed)
        st["out"] = torch.empty_like(st["r"])
    else:
        st["q"] = torch.from_numpy(np.ascontiguousarray(_state(case, s.coords(), T, inf, seed))).cuda()
        st["out"] = torch.empty_like(st["q"])
    torch.cuda.synchronize()
    if kind == "cycles":   # the first implicit stage of a step from this state
        dt = {"vortex": 0.1, "cylinder": 0.05, "sphere": 0.1, "ellipse": 0.01}[case["flow"]]
        pmgfr.pmg_residual(s.h, 0, st["q"], st["out"])
        src = (_cons(st["q"]) + OMEGA * dt * st["out"]) / (OMEGA * dt)
        torch.cuda.synchronize()
        pmgfr.pmg_set_stage(s.h, src, OMEGA * dt)
        st["dtau"] = 0.01 if case["flow"] == "vortex" else 1e-3
    if kind == "step" and case["solver"] == "nk":
        pmgfr.pmg_set_stage_solver(s.h, pmgfr.PMG_STAGE_NK, krylov_dim=30, max_krylov=60, dtau_pc=10.0, pc_refresh=2,
                                   state_scale=(T, 1.0, 1.0, T))
    return st


def run(st):
    s, out = st["s"], st["out"]
    if st["kind"] == "residual":
        return pmgfr.pmg_residual(s.h, 0, st["q"], out)
    if st["kind"] == "blocks":
        pmgfr.pmg_set_blocks(s.h, 0, st["D"])
        pmgfr.pmg_factor_blocks(s.h, 0)
        return pmgfr.pmg_apply_blocks(s.h, 0, st["r"], out)
    pmgfr.pmg_set_state(s.h, 0, st["q"])
    if st["kind"] == "cycles":
        for k in range(10):
            pmgfr.pmg_vcycle(s.h, st["dtau"], refresh=k == 0)
    else:
        pmgfr.pmg_esdirk_step(s.h, 0.1)
    return pmgfr.pmg_get_state(s.h, 0, out)


# ------------------------------------------------------------------ work
def _residual_work(dim, E, P, visc):
    """Bytes (state in, residual out, metrics, face geometry) and operations of one residual."""
    n1, nv = P + 1, dim + 2
    N, F = n1 ** dim, dim * E * n1 ** (dim - 1)   # F: face points, each face once
    nbytes = 8 * (E * N * (2 * nv + dim * dim + 1) + F * (dim + 1))
    face = 2 * 2 * nv * n1 + (190 if dim == 2 else 235)
    point = dim * (10 + 4 * nv) + nv * dim * (2 * n1 + 8)
    if visc:
        g = dim * (dim + 1)
        face += 2 * 2 * g * n1 + 60
        point += 2 * ((dim + 1) * dim * (2 * n1 + 2 * dim)) + 60
    return nbytes, F * face + E * N * point


def work(case):
    levels = [int(p) for p in case["levels"].split("-")]
    flow = case["flow"]
    dim = 2 if flow in ("vortex", "cylinder") else 3
    E = {"vortex": case["a"] * case["b"], "cylinder": case["a"] * case["b"], "sphere": 6 * case["a"] ** 2 * case["b"],
         "ellipse": case["a"] * case["b"] * case["c"], "box3": case["a"] * case["b"] * case["c"]}[flow]
    visc = flow in ("cylinder", "ellipse")
    n = [(dim + 2) * (P + 1) ** dim for P in levels]
    if case["kind"] == "residual":
        nbytes, flops = _residual_work(dim, E, levels[0], visc)
        return dict(bytes=nbytes, flops=flops)
    wb = {"fp64": 8, "fp32": 4, "bf16": 2}[case["blocks"]]
    if case["kind"] == "blocks":
        return dict(bytes=E * (8 * n[0] ** 2 + 16 * n[0]), flops=E * (2 * n[0] ** 3 + 2 * n[0] ** 2))
    # V-cycles and rebuilds of the pass; a step takes about so many (measured): 800 pseudo-iterations and 6
    # rebuilds, or 76 preconditioner cycles and 6 rebuilds
    cycles, rebuilds = (10, 1) if case["kind"] == "cycles" else (800, 6) if case["solver"] == "ptc" else (76, 6)
    nbytes, flops = 16 * E * n[0], 0
    for l, P in enumerate(levels):
        sweeps = SMOOTH[l] * (1 if l == len(levels) - 1 else 2)
        rb, rf = _residual_work(dim, E, P, visc)
        blk = E * n[l] ** 2 * wb
        big = blk + rb > 129e6   # a level beyond the L2 cache is read by every sweep, another once a cycle
        nbytes += cycles * (sweeps if big else 1) * (blk + rb)
        flops += cycles * sweeps * (rf + 2 * E * n[l] ** 2) + rebuilds * 2 * E * n[l] ** 3
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ values in 64 bits
def exact(case, seed):
    """The residual and the blocks' solution by plain numpy and torch in 64
    bits; the cycles and steps would take minutes that way."""
    if case["kind"] == "blocks":
        D, r = _own_blocks(case, seed)
        E, N = r.shape[1:]
        x = torch.linalg.solve(D, r.permute(1, 0, 2).reshape(E, -1, 1))
        return x.reshape(E, 5, N).permute(1, 0, 2).contiguous()
    if case["kind"] != "residual":
        return None
    nodes, nbr, dim, levels, T, inf, kw = _setup(case)
    fr = _FR(nodes, nbr, dim, levels[0], kw.get("mu", 0.0), T, inf,
             kw.get("kappa", 0.0) * kw["Ma_inf"] if kw.get("cutoff") else 0.0)
    return fr.residual(_state(case, fr.xyz, T, inf, seed))


def _lagrange(x, t):
    """Values [t, k] and derivatives of the Lagrange basis on x."""
    n = len(x)
    V, dV = np.ones((len(t), n)), np.zeros((len(t), n))
    for k in range(n):
        for m in range(n):
            if m != k:
                dV[:, k] = dV[:, k] * (t - x[m]) / (x[k] - x[m]) + V[:, k] / (x[k] - x[m])
                V[:, k] *= (t - x[m]) / (x[k] - x[m])
    return V, dV


class _FR:
    """The flux-reconstruction residual on one mesh.  Fields are arrays
    (..., E, [k,] j, i); axis -1 is the first reference direction."""

    def __init__(self, nodes, nbr, dim, P, mu, T0, inf, eps_min):
        self.dim, self.P, self.n1, self.mu, self.p0, self.inf, self.eps_min = dim, P, P + 1, mu, T0, inf, eps_min
        self.x, w = np.polynomial.legendre.leggauss(P + 1)
        self.D = _lagrange(self.x, self.x)[1]
        ends = _lagrange(self.x, np.array([-1.0, 1.0]))[0]
        self.end = ends                                             # traces at -1 and +1
        self.g = np.stack([-ends[0] / w, ends[1] / w])              # derivatives of the DG correction functions
        E = nodes.shape[0]
        self.E, self.N, self.NF = E, (P + 1) ** dim, (P + 1) ** (dim - 1)
        ng = round(nodes.shape[1] ** (1.0 / dim))
        X = nodes.transpose(2, 0, 1).reshape((dim, E) + (ng,) * dim)
        self.X, self.gx = X, np.linspace(-1.0, 1.0, ng)
        # faces as (direction, side); quadrilaterals number them 0: eta-, 1: xi+, 2: eta+, 3: xi-
        self.faces = [(1, 0), (0, 1), (1, 1), (0, 0)] if dim == 2 else [(f // 2, f % 2) for f in range(6)]
        self.en, self.fn = nbr[:, :, 0], nbr[:, :, 1]
        o, P1 = nbr[:, :, 2], np.arange(P + 1)
        if dim == 2:
            self.fp2 = np.where(o[:, :, None] != 0, P - P1, P1)
        else:
            b, a = (t.reshape(-1) for t in np.meshgrid(P1, P1, indexing="ij"))
            o = o[:, :, None]
            s, t = np.where(o & 4, b, a), np.where(o & 4, a, b)
            self.fp2 = np.where(o & 2, P - t, t) * (P + 1) + np.where(o & 1, P - s, s)
        pts = [self.x] * dim
        self.xyz = self._map(pts)[0].reshape(dim, E, -1).transpose(1, 2, 0)
        self.Ja, J = self._metric(pts)                              # Ja[i][n], |J|
        self.iJ = 1.0 / J
        nrm, self.iJf = [], []
        for d, s in self.faces:
            p = list(pts)
            p[d] = np.array([2.0 * s - 1.0])
            Ja, J = self._metric(p)
            nrm.append((2.0 * s - 1.0) * Ja[d].reshape(dim, E, -1))
            self.iJf.append(1.0 / J.reshape(E, -1))
        nrm = np.stack(nrm, 2)                                      # (dim, E, face, point)
        self.dS = np.sqrt((nrm ** 2).sum(0))
        self.nrm = nrm / self.dS
        self.iJf = np.stack(self.iJf, 1)

    def _along(self, A, F, d):
        """Matrix A along reference direction d of F."""
        return np.moveaxis(np.tensordot(F, A, axes=([F.ndim - 1 - d], [1])), -1, F.ndim - 1 - d)

    def _map(self, pts, F=None, gx=None):
        """An interpolant on gx and its reference derivatives at a tensor grid of points."""
        F, gx = self.X if F is None else F, self.gx if gx is None else gx
        L = [_lagrange(gx, p) for p in pts]
        out = []
        for k in [None] + list(range(self.dim)):
            G = F
            for d in range(self.dim):
                G = self._along(L[d][1 if k == d else 0], G, d)
            out.append(G)
        return out[0], out[1:]

    def _metric(self, pts):
        X, dX = self._map(pts)
        if self.dim == 2:
            (xx, yx), (xe, ye) = dX
            return np.array([[ye, -xe], [-yx, xx]]), xx * ye - xe * yx
        J = (np.cross(dX[0], dX[1], axis=0) * dX[2]).sum(0)
        # conservative curl form on Gauss-Lobatto points of degree max(P, geometry order)
        n = max(self.P, len(self.gx) - 1, 1)
        c = np.zeros(n + 1)
        c[n] = 1.0
        gl = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c)).real),
                             [1.0]]) if n > 1 else np.array([-1.0, 1.0])
        Y, dY = self._map([gl] * 3)
        Ja = np.zeros((3, 3) + J.shape)
        for c in range(3):
            m, l = (c + 1) % 3, (c + 2) % 3
            dW = [self._map(pts, Y[l] * dY[k][m], gl)[1] for k in range(3)]   # dW[k][j] = d_j W_k
            for i in range(3):
                j, k = (i + 1) % 3, (i + 2) % 3
                Ja[i, c] = -(dW[k][j] - dW[j][k])
        return Ja, J

    def _trace(self, F):
        """Traces (..., E, face, point) of a field (..., E, [k,] j, i)."""
        out = []
        for d, s in self.faces:
            out.append(np.tensordot(F, self.end[s], axes=([F.ndim - 1 - d], [0])).reshape(F.shape[:-self.dim] + (-1,)))
        return np.stack(out, -2)

    def _other(self, T):
        """The neighbour's values of a trace (garbage on boundary faces)."""
        return T[..., np.maximum(self.en, 0)[:, :, None], np.where(self.en < 0, 0, self.fn)[:, :, None], self.fp2]

    def _correct(self, F, jump, d):
        """Derivative of F along d plus the correction of its jumps (..., E, face, point) on that direction's faces."""
        out = self._along(self.D, F, d)
        for f, (fd, s) in enumerate(self.faces):
            if fd == d:
                sh = list(F.shape)
                ax = len(sh) - 1 - d
                sh[ax] = 1
                gs = [1] * len(sh)
                gs[ax] = self.n1
                out = out + jump[..., f, :].reshape(sh) * self.g[s].reshape(gs)
        return out

    def _flux(self, q, pg):
        """Inviscid fluxes [direction][variable] of (p, velocity, T); pg is the pressure of the momentum flux."""
        rho, vel = q[0] / q[-1], q[1:-1]
        H = GAMMA / (GAMMA - 1.0) * q[-1] + 0.5 * (vel ** 2).sum(0)
        return np.array([[rho * vel[c]] + [rho * vel[c] * vel[k] + (pg if k == c else 0.0) for k in range(self.dim)] +
                         [rho * vel[c] * H] for c in range(self.dim)])

    def _viscous(self, vel, G):
        """Viscous fluxes [direction][momentum rows, energy]; G[c][k] = d(velocity, T)_k / dx_c."""
        d = self.dim
        div = sum(G[c, c] for c in range(d))
        tau = self.mu * (G[:, :d] + G[:, :d].swapaxes(0, 1))
        for c in range(d):
            tau[c, c] -= self.mu * 2.0 / 3.0 * div
        heat = self.mu * GAMMA / (GAMMA - 1.0) / PR
        return np.concatenate([tau, ((tau * vel).sum(1) + heat * G[:, d])[:, None]], 1)

    def _roe(self, qm, qp, dq, pm, pp):
        """Central flux minus half of Gamma |Gamma^-1 A_n| dq at the mean state, through dS."""
        n, d = self.nrm, self.dim
        f = 0.5 * ((self._flux(qm, pm) + self._flux(qp, pp)) * n[:, None]).sum(0)
        q = 0.5 * (qm + qp)
        p, vel, T = q[0], q[1:-1], q[-1]
        rho, c2, Cp = p / T, GAMMA * T, GAMMA / (GAMMA - 1.0)
        vv, un = (vel ** 2).sum(0), (vel * n).sum(0)
        e2 = np.minimum(1.0, np.maximum(self.eps_min ** 2, vv / c2))
        dp, dun, dT = dq[0], (dq[1:-1] * n).sum(0), dq[-1]
        # Gamma^-1 A_n on (p, u_n): [[e2 u, rho e2 c2], [1/rho, u]]; T: (T row) with eigenvalue u_n
        B = np.array([[e2 * un, rho * e2 * c2], [1.0 / rho, un]])
        h = 0.5 * (1.0 + e2) * un
        cp = np.sqrt((0.5 * (1.0 - e2) * un) ** 2 + e2 * c2)
        l1, l2, lu = np.abs(h + cp), np.abs(h - cp), np.abs(un)
        a1 = (l1 - l2) / (2.0 * cp)
        a0 = l1 - a1 * (h + cp)
        z = np.array([a0 * dp + a1 * (B[0, 0] * dp + B[0, 1] * dun), a0 * dun + a1 * (B[1, 0] * dp + B[1, 1] * dun)])
        # the T row r = (-(1 - e2) u_n / (rho Cp), e2 (gamma - 1) T) times (|B| - |u_n|) (B - u_n)^-1
        w = np.array([rho * dun, (dp / rho + (1.0 - e2) * un * dun) / (e2 * c2)])
        y = np.array([(a0 - lu) * w[0] + a1 * (B[0, 0] * w[0] + B[0, 1] * w[1]),
                      (a0 - lu) * w[1] + a1 * (B[1, 0] * w[0] + B[1, 1] * w[1])])
        xT = -(1.0 - e2) * un / (rho * Cp) * y[0] + e2 * (GAMMA - 1.0) * T * y[1] + lu * dT
        xv = z[1] * n + lu * (dq[1:-1] - dun * n)
        # Gamma = M K, K the identity but for K_pp = 1/e2 and K_Tp = (1/e2 - 1)/(rho Cp)
        yp, yT = z[0] / e2, (1.0 / e2 - 1.0) / (rho * Cp) * z[0] + xT
        drho = (yp - rho * yT) / T
        diss = np.concatenate([[drho], vel * drho + rho * xv,
                               [(Cp * T + 0.5 * vv) * drho - yp + rho * (vel * xv).sum(0) + rho * Cp * yT]])
        return (f - 0.5 * diss) * self.dS

    def residual(self, q):
        d, nv = self.dim, self.dim + 2
        shape = q.shape
        q = q.reshape((nv, self.E) + (self.n1,) * d)
        base = np.zeros(nv)
        base[0] = base[-1] = self.p0
        dev = q - base.reshape((nv,) + (1,) * (q.ndim - 1))         # p and T relative to the free stream
        tm = self._trace(dev)
        tp = self._other(tm)
        bnd = (self.en < 0)[:, :, None]
        if self.inf is not None:
            far, slip = bnd & (self.fn == W.BC_FARFIELD)[:, :, None], bnd & (self.fn == W.BC_SLIP_WALL)[:, :, None]
            ghost = tm.copy()
            ghost[1:-1] = np.where(slip, tm[1:-1] - 2.0 * (tm[1:-1] * self.nrm).sum(0) * self.nrm, -tm[1:-1])
            ghost = np.where(far, (np.array(self.inf) - base).reshape(-1, 1, 1, 1), ghost)
            tp = np.where(bnd, ghost, tp)
        b4 = base.reshape(-1, 1, 1, 1)
        com = self._roe(tm + b4, tp + b4, tp - tm, tm[0], tp[0])
        fl = self._flux(q, dev[0])
        if self.mu:
            gv = [self._along(self.D, dev[1:], k) for k in range(d)]
            brk = self.iJ * np.array([sum(self.Ja[k, c] * gv[k] for k in range(d)) for c in range(d)])
            jump = 0.5 * (tp - tm)[1:]
            gv = [self._correct(dev[1:], jump, k) for k in range(d)]
            cor = self.iJ * np.array([sum(self.Ja[k, c] * gv[k] for k in range(d)) for c in range(d)])
            fl[:, 1:] -= self._viscous(q[1:-1], cor)
            gm = self._trace(brk)
            gp = np.where(bnd, gm, self._other(gm))
            iJp = np.where(bnd, self.iJf, self._other(self.iJf))
            lift = 0.25 * 2.0 * self.n1 ** 2 * (self.iJf + iJp) * self.dS * self.nrm
            fv = (self._viscous(0.5 * (tm + tp)[1:-1], 0.5 * (gm + gp) + lift[:, None] * (tp - tm)[None, 1:]) *
                  self.nrm[:, None]).sum(0) * self.dS
            fv[-1] = np.where(bnd & (self.fn != W.BC_FARFIELD)[:, :, None], 0.0, fv[-1])
            com[1:] -= fv
        side = np.array([2.0 * s - 1.0 for _, s in self.faces]).reshape(-1, 1)
        div = 0.0
        for k in range(d):
            F = sum(self.Ja[k, c] * fl[c] for c in range(d))
            div = div + self._correct(F, side * com - self._trace(F), k)
        return np.ascontiguousarray((-div * self.iJ).reshape(shape))

"""Fused P = 0 sweeps of hexahedra (k3_fused.cu: one launch per sweep, the six
face fluxes of an element formed in the sweep) against the general path (face
fluxes, then the volume kernel) on the same problem, at element counts that
leave the last warp one to four elements (it takes five), with every boundary
type, relative element rotation and block precision.

Both sum the same terms, in another order, so residuals differ by their FP64
rounding.  With FP64 blocks the two V-cycles agree to 1e-8 of the change they
make, the bound of the other V-cycle tests; FP32 and BF16 blocks take residuals
rounded to FP32 (6e-8), where last-bit differences become one FP32 rounding, and
eight sweeps of n = 5 rows add up to 40 of them: 1e-5.
"""
import numpy as np
import pytest

from paper_1908_03972_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_03972_gb300 import build, pmgfr
    build.build()
    pmgfr.load()


def _channel(**kw):
    nodes, nbr = W.channel(3, 2, Ng=1, **kw)
    return W.extrude(nodes, nbr, 1, nz=1, z0=0.0, z1=2.0)


MESHES = {
    "rotated": lambda: (W.periodic_box3d(3, 2, 3, Ng=1, rotations={1: 7, 8: 14, 12: 21, 17: 3}), 1),
    "curved": lambda: (W.periodic_box3d(3, 3, 3, Ng=2, perturb=0.3, rotations={0: 5, 4: 11, 26: 17}), 2),
    "noslip_farfield": lambda: (_channel(top=W.BC_FARFIELD), 1),
    "slip_farfield": lambda: (_channel(bottom=W.BC_SLIP_WALL, top=W.BC_FARFIELD), 1),   # slip walls need mu = 0
    "shell": lambda: (W.cubed_sphere_shell(2, 1, 0.5, 2.0, Ng=2, wall=W.BC_FARFIELD), 2),
}


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("name,mu", [(n, m) for n in MESHES for m in (0.0, 0.02) if n != "slip_farfield" or m == 0.0])
def test_fused_sweep3_matches_split_sweep(monkeypatch, name, mu, prec):
    from paper_1908_03972_gb300 import pmgfr
    (nodes, nbr), Ng = MESHES[name]()
    Ma = 0.2
    T = W.freestream_T(Ma, speed=1.0)
    out = []
    for fuse in (None, "-1"):
        monkeypatch.delenv("PMG_FUSE_MAX_P", raising=False)
        if fuse:
            monkeypatch.setenv("PMG_FUSE_MAX_P", fuse)
        gpu = pmgfr.Solver(nodes, nbr, [1, 0], [1, 8], dim=3, mu=mu, Ma_inf=Ma, block_prec=prec, cutoff=1, kappa=1.0,
                           q_inf3=(T, 1.0, 0.0, 0.0, T))
        try:
            x = gpu.coords(0)
            q = W.uniform_state3(x.shape[0], x.shape[1], T, 1.0, 0.2, -0.1, T)
            q = q * (1 + 1e-2 * np.random.default_rng(3).standard_normal(q.shape))
            gpu.set_stage(np.zeros_like(q), 0.05)
            out.append(gpu.vcycle(q, 0.5)[0])
        finally:
            gpu.close()
    for v in range(5):
        change = np.abs(out[1][v] - q[v]).max()
        assert change > 0
        assert np.abs(out[0][v] - out[1][v]).max() <= (1e-8 if prec == 0 else 1e-5) * change, v

"""Block assembly (k_assemble.cu) against the oracle's complex-step blocks where
tests/test_gpu_assemble.py does not go: hexahedra at P = 3 (n = 320) on curved
elements with rotated local axes, hexahedra between a no-slip wall and a far field
on elements curved in the plane of the wall's normal, and 121 quadrilaterals, which
no number of elements a CTA takes divides at any order.  Inviscid and viscous; the
bound of the other block tests, 1e-10 relative Frobenius per element.
"""
import numpy as np
import pytest

import oracle as O
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


def _compare(orc, gpu, q):
    q = q * (1 + 1e-2 * np.random.default_rng(5).standard_normal(q.shape))
    orc.set_stage(np.zeros_like(q), 0.05)
    gpu.set_stage(np.zeros_like(q), 0.05)
    Do, Dg = orc.blocks(q, 0.7), gpu.blocks(q, 0.7)
    for e in range(orc.E):
        assert np.linalg.norm(Dg[e] - Do[e]) <= 1e-10 * np.linalg.norm(Do[e]), e


@pytest.mark.parametrize("mu", [0.0, 0.02])
def test_curved_rotated_hexahedra_at_p3(mu):
    from paper_1908_03972_gb300 import pmgfr
    kw = dict(Ma_inf=0.3, mu=mu)
    nodes, nbr = W.periodic_box3d(3, 3, 2, Ng=2, perturb=0.3, rotations={0: 5, 4: 11, 13: 17, 17: 3})
    orc = O.Oracle3(nodes, nbr, 2, [3], [1], **kw)
    gpu = pmgfr.Solver(nodes, nbr, [3], [1], dim=3, **kw)
    try:
        _compare(orc, gpu, W.vortex3d(orc.coords(), Ma_inf=0.3, center=(4.0, 6.0)))
    finally:
        gpu.close()


@pytest.mark.parametrize("mu", [0.0, 0.02])
@pytest.mark.parametrize("P", [0, 1, 2, 3])
def test_hexahedra_between_a_wall_and_a_far_field(P, mu):
    from paper_1908_03972_gb300 import pmgfr
    Ma = 0.2
    T = W.freestream_T(Ma, speed=1.0)
    inf = (T, 1.0, 0.0, 0.0, T)
    nodes, nbr = W.extrude(*W.channel(3, 2, Ng=2, perturb=0.3, top=W.BC_FARFIELD), 2, nz=1, z0=0.0, z1=2.0)
    orc = O.Oracle3(nodes, nbr, 2, [P], [1], Ma_inf=Ma, mu=mu, cutoff=1, kappa=1.0, q_inf=inf)
    gpu = pmgfr.Solver(nodes, nbr, [P], [1], dim=3, Ma_inf=Ma, mu=mu, cutoff=1, kappa=1.0, q_inf3=inf)
    try:
        x = orc.coords()
        _compare(orc, gpu, W.uniform_state3(x.shape[0], x.shape[1], T, 1.0, 0.2, -0.1, T))
    finally:
        gpu.close()


@pytest.mark.parametrize("mu", [0.0, 0.02])
@pytest.mark.parametrize("P", [0, 1, 2, 3, 4, 5])
def test_quadrilaterals_with_a_part_empty_cta_at_every_order(P, mu):
    from paper_1908_03972_gb300 import pmgfr
    kw = dict(Ma_inf=0.3, mu=mu)
    nodes, nbr = W.flip_elements(*W.periodic_box(11, 11, Ng=2, perturb=0.3), [0, 17, 120], 2)
    orc = O.Oracle(nodes, nbr, 2, [P], [1], **kw)
    assert all(orc.E % k for k in (3, 4, 5, 7, 8, 10, 16, 32))   # elements per CTA of both kernels, all orders
    gpu = pmgfr.Solver(nodes, nbr, [P], [1], **kw)
    try:
        _compare(orc, gpu, W.isentropic_vortex(orc.coords(), Ma_inf=0.3, center=(4.0, 6.0)))
    finally:
        gpu.close()

"""Block assembly (k_assemble.cu) against the oracle's complex-step blocks at
every order, with element counts that leave the last CTA part empty for every
number of elements a CTA takes (35 quadrilaterals, 27 hexahedra), inviscid and
viscous, on curved meshes with renumbered elements; the bound is that of the
other block tests, 1e-10 relative Frobenius per element.
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


@pytest.mark.parametrize("mu", [0.0, 0.02])
@pytest.mark.parametrize("dim,P", [(2, 0), (2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (3, 0), (3, 1), (3, 2)])
def test_assembled_blocks_with_part_empty_ctas(dim, P, mu):
    from paper_1908_03972_gb300 import pmgfr
    kw = dict(Ma_inf=0.3, mu=mu)
    if dim == 2:
        nodes, nbr = W.flip_elements(*W.periodic_box(7, 5, Ng=2, perturb=0.3), [0, 8, 34], 2)
        orc = O.Oracle(nodes, nbr, 2, [P], [1], **kw)
    else:
        nodes, nbr = W.periodic_box3d(3, 3, 3, Ng=2, perturb=0.3, rotations={0: 5, 4: 11, 13: 17, 26: 3})
        orc = O.Oracle3(nodes, nbr, 2, [P], [1], **kw)
    gpu = pmgfr.Solver(nodes, nbr, [P], [1], dim=dim, **kw)
    try:
        xyz = orc.coords()
        q = (W.isentropic_vortex(xyz, Ma_inf=0.3, center=(4.0, 6.0)) if dim == 2
             else W.vortex3d(xyz, Ma_inf=0.3, center=(4.0, 6.0)))
        q = q * (1 + 1e-2 * np.random.default_rng(5).standard_normal(q.shape))
        orc.set_stage(np.zeros_like(q), 0.05)
        gpu.set_stage(np.zeros_like(q), 0.05)
        Do, Dg = orc.blocks(q, 0.7), gpu.blocks(q, 0.7)
        for e in range(orc.E):
            assert np.linalg.norm(Dg[e] - Do[e]) <= 1e-10 * np.linalg.norm(Do[e]), e
    finally:
        gpu.close()

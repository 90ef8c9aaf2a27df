"""Several viscous sweeps in a row against the oracle: from the second on, the
broken gradients come from the update of the sweep before (k_residual.cu,
k3_residual.cu) instead of a gradient launch, and so do those of the residual
after the last one.  Element counts leave the last CTA part empty (35
quadrilaterals, 27 hexahedra); the bound is that of the other V-cycle tests with
FP64 blocks and fluxes, 1e-8 of the change.
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


@pytest.mark.parametrize("levels", [[0], [1], [2], [3], [4], [5], [3, 1]])
@pytest.mark.parametrize("dim", [2, 3])
def test_sweeps_reuse_gradients(dim, levels):
    from paper_1908_03972_gb300 import pmgfr
    if dim == 3 and levels[0] > 3:
        pytest.skip("hexahedra have P <= 3")
    kw = dict(Ma_inf=0.2, mu=0.02)
    smooth = [3, 4][:len(levels)]
    if dim == 2:
        nodes, nbr = W.flip_elements(*W.periodic_box(7, 5, Ng=2, perturb=0.3), [0, 8, 34], 2)
        orc = O.Oracle(nodes, nbr, 2, levels, smooth, **kw)
    else:
        nodes, nbr = W.periodic_box3d(3, 3, 3, Ng=2, perturb=0.3, rotations={0: 5, 4: 11, 13: 17, 26: 3})
        orc = O.Oracle3(nodes, nbr, 2, levels, smooth, **kw)
    gpu = pmgfr.Solver(nodes, nbr, levels, smooth, dim=dim, flux_prec=pmgfr.PMG_FLUX_FP64, **kw)
    try:
        xyz = orc.coords()
        q = (W.isentropic_vortex(xyz, Ma_inf=0.2, center=(4.0, 6.0)) if dim == 2
             else W.vortex3d(xyz, Ma_inf=0.2, center=(4.0, 6.0)))
        rho, u = q[0] / q[-1], q[1:-1]
        qc = np.concatenate([rho[None], rho * u, (rho * (q[-1] / 0.4 + 0.5 * (u * u).sum(0)))[None]])
        src = qc / 0.05 + 0.5 * orc.residual(q)
        orc.set_stage(src, 0.05)
        gpu.set_stage(src, 0.05)
        qo = orc.vcycle(q, 0.7, refresh=True)
        qg, _ = gpu.vcycle(q, 0.7, refresh=True)
        change = np.abs(qo - q).max(axis=(1, 2))
        assert (np.abs(qg - qo).max(axis=(1, 2)) <= 1e-8 * np.maximum(change, change.max() * 1e-3)).all()
    finally:
        gpu.close()

"""Viscous sweeps whose update leaves the broken gradients for the next one, in
place of those it read (k_residual.cu), against the oracle, on 121
quadrilaterals: no number of elements that a CTA of the gradient, residual or
update launches takes divides it, so the last CTA is part empty (the updates of
so few elements at P = 5 take one to a CTA; tests/test_gpu_few_elements.py has
three).  FP64 blocks and fluxes; the bound is that of the other V-cycle tests,
1e-8 of the change.
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


@pytest.mark.parametrize("P", [1, 2, 3, 4, 5])
def test_gradients_left_by_the_update_in_a_part_empty_cta(P):
    from paper_1908_03972_gb300 import pmgfr
    nodes, nbr = W.flip_elements(*W.periodic_box(11, 11, Ng=2, perturb=0.3), [0, 17, 120], 2)
    kw = dict(Ma_inf=0.2, mu=0.02)
    orc = O.Oracle(nodes, nbr, 2, [P], [3], **kw)
    assert all(orc.E % k for k in (3, 4, 5, 7, 8, 14, 32))   # elements per CTA of the launches, all orders
    gpu = pmgfr.Solver(nodes, nbr, [P], [3], flux_prec=pmgfr.PMG_FLUX_FP64, **kw)
    try:
        q = W.isentropic_vortex(orc.coords(), Ma_inf=0.2, center=(4.0, 6.0))
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

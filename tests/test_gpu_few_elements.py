"""Sweeps at P = 4 and 5 on both sides of the rule for elements per CTA
(sweep_common.cuh: two and one on few elements, five and three on many) against
the oracle, with a part-empty last CTA wherever a CTA takes more than one: 121 and
1221 quadrilaterals at P = 4, 121 and 154 at P = 5, viscous, inviscid and
inviscid in double-word with gauge storage.

FP64 blocks; 1e-8 of the change, the bound of the other V-cycle tests, and with
double-word fluxes (about 2^-44 where binary64 has 2^-53) 2^9 times that.
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


@pytest.mark.parametrize("mode", ["viscous", "inviscid", "double-word"])
@pytest.mark.parametrize("P,a,b", [(4, 11, 11), (4, 37, 33), (5, 11, 11), (5, 14, 11)])
def test_sweeps_on_both_sides_of_the_rule(P, a, b, mode):
    from paper_1908_03972_gb300 import pmgfr
    nodes, nbr = W.flip_elements(*W.periodic_box(a, b, Ng=2, perturb=0.3), [0, 17, a * b - 1], 2)
    kw = dict(Ma_inf=0.2, mu=0.02 if mode == "viscous" else 0.0)
    orc = O.Oracle(nodes, nbr, 2, [P], [3], **kw)
    dword = mode == "double-word"
    gpu = pmgfr.Solver(nodes, nbr, [P], [3], flux_prec=pmgfr.PMG_FLUX_DW_SMOOTH if dword else pmgfr.PMG_FLUX_FP64,
                       p_gauge=W.freestream_T(0.2) if dword else 0.0, **kw)
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
        tol = 1e-8 * (512 if dword else 1)
        assert (np.abs(qg - qo).max(axis=(1, 2)) <= tol * np.maximum(change, change.max() * 1e-3)).all()
    finally:
        gpu.close()

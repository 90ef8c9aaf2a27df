"""The double-word Roe flux (physics_dw.cuh) over the Mach numbers its FP32 range
allows: the residual under PMG_FLUX_DW against PMG_FLUX_FP64 on the same state.
p and T are about 1/Ma^2 at unit speed, so at Ma = 1e-10 a product of the two
would pass 2^127 while each alone is far from it.

Bound: the face flux is off by at most 64 u^2 (u = 2^-24) of its row's scale
(rho |u|, rho |u|^2, rho |u| H; its longest chain has fewer than twenty
operations of at most 6.5 u^2, most of them on terms below the scale), and a
point of an element of side h takes four face fluxes with weights of at most
(P+1)^2 / 2 times dS / |J| = 2 / h.
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


@pytest.mark.parametrize("Ma", [1e-3, 1e-6, 1e-8, 1e-9, 1e-10])
def test_double_word_flux_at_low_mach_numbers(Ma):
    from paper_1908_03972_gb300 import pmgfr
    P, n = 2, 6
    nodes, nbr = W.periodic_box(n, n, Ng=1)
    T = W.freestream_T(Ma, speed=1.0)
    out = []
    for flux in (pmgfr.PMG_FLUX_DW, pmgfr.PMG_FLUX_FP64):
        s = pmgfr.Solver(nodes, nbr, [P], [1], Ma_inf=Ma, p_gauge=T, flux_prec=flux)
        try:
            x = s.coords()
            ph = 2.0 * np.pi / 10.0 * x
            q = np.stack([np.full(x.shape[:2], T), 1.0 + 0.2 * np.sin(ph[..., 1]), 0.3 * np.cos(ph[..., 0]),
                          np.full(x.shape[:2], T)])
            out.append(s.residual(q))
        finally:
            s.close()
    speed = 1.3
    amp = 4 * (P + 1) ** 2 / 2 * 2 / (10.0 / n)
    scale = np.array([speed, speed ** 2, speed ** 2, speed * 3.5 * T])
    assert np.isfinite(out[0]).all()
    err = np.abs(out[0] - out[1]).max(axis=(1, 2))
    assert (err <= 64 * 2.0 ** -48 * amp * scale).all(), err / scale

"""One-launch sweeps on the finest level with FP32 and BF16 blocks against the face
and volume launches (PMG_FUSE_MAX_P = -1), two V-cycles on 121 quadrilaterals (a
part-empty last CTA on both sides at every order).

Both sides take residuals whose last bits differ to the same FP32 products, so what
differs is FP32 roundings of residual entries (6e-8 of an entry): a V-cycle of the
longest hierarchy here has 14 sweeps, each of at most n = 36 rows, hence at most
2 x 14 x 36 x 6e-8 = 6e-5 of the change.
"""
import numpy as np
import pytest

from paper_1908_03972_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MA = 0.05


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_03972_gb300 import build, pmgfr
    build.build()
    pmgfr.load()


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("flux,gauge", [("fp64", False), ("fp64", True), ("dw", False), ("dw", True)])
@pytest.mark.parametrize("levels,smooth", [([2, 1, 0], [2, 3, 4]), ([1, 0], [3, 2]), ([0], [3])])
def test_fused_finest_sweeps_in_fp32(monkeypatch, levels, smooth, flux, gauge, prec):
    from paper_1908_03972_gb300 import pmgfr
    nodes, nbr = W.flip_elements(*W.periodic_box(11, 11, Ng=1), [0, 17, 120], 1)
    out = []
    for fuse in (None, "-1"):
        monkeypatch.delenv("PMG_FUSE_MAX_P", raising=False)
        if fuse:
            monkeypatch.setenv("PMG_FUSE_MAX_P", fuse)
        gpu = pmgfr.Solver(nodes, nbr, levels, smooth, Ma_inf=MA, block_prec=prec,
                           p_gauge=W.freestream_T(MA) if gauge else 0.0,
                           flux_prec=pmgfr.PMG_FLUX_FP64 if flux == "fp64" else pmgfr.PMG_FLUX_DW_SMOOTH)
        try:
            q = W.isentropic_vortex(gpu.coords(), Ma_inf=MA, center=(4.0, 6.0))
            src = gpu.residual(q)
            rho = q[0] / q[3]
            qc = np.stack([rho, rho * q[1], rho * q[2], rho * (q[3] / 0.4 + 0.5 * (q[1] ** 2 + q[2] ** 2))])
            gpu.set_stage(qc / 0.05 + src, 0.05)
            q1, _ = gpu.vcycle(q, 0.7)
            q2, _ = gpu.vcycle(q1, 0.7, refresh=False)
            out.append((q1, q2))
        finally:
            gpu.close()
    for k in (0, 1):
        change = np.abs(out[1][k] - q).max(axis=(1, 2))
        assert (change > 0).all()
        assert (np.abs(out[0][k] - out[1][k]).max(axis=(1, 2)) <= 6e-5 * change).all(), k

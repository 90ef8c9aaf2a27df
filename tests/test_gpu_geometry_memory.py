"""Metrics and face geometry are held in double-word, next to binary64, only by
contexts whose sweeps read them so (quadrilaterals, gauge storage, mu = 0, a
double-word flux_prec): the device memory of the others is smaller by that copy.
"""
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


def _used(nodes, nbr, **kw):
    import torch
    from paper_1908_03972_gb300 import pmgfr
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    s = pmgfr.Solver(nodes, nbr, [1], [1], block_prec=1, Ma_inf=0.1, **kw)
    try:
        torch.cuda.synchronize()
        return free0 - torch.cuda.mem_get_info()[0]
    finally:
        s.close()


def test_only_double_word_sweeps_hold_double_word_geometry():
    from paper_1908_03972_gb300 import pmgfr
    n = 300
    nodes, nbr = W.periodic_box(n, n, Ng=1)
    T = W.freestream_T(0.1)
    words = 8 * n * n * (4 * 5 + 4 * 2 * 3)            # 5 metrics a point, 3 numbers a face point
    dw = _used(nodes, nbr, p_gauge=T, flux_prec=pmgfr.PMG_FLUX_DW_SMOOTH)
    slack = 6 << 20                                    # rounding of the allocations
    for kw in (dict(p_gauge=T, flux_prec=pmgfr.PMG_FLUX_FP64), dict(p_gauge=0.0)):
        other = _used(nodes, nbr, **kw)
        assert abs(dw - other - words) <= slack, (kw, dw, other, words)

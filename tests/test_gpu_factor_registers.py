"""The register factorisation (k_factor.cu) against the column-by-column one
(k_factor_cluster.cu, PMG_FACTOR_CLUSTER = 8) at every block size and
precision of the library: both do the same operations on every entry, so the
factored blocks applied to a vector agree bit for bit.  The blocks: random
ones, one full of equal pivot candidates (the tie rule: the first row under
the interchanges), one whose rows and columns span 24 decades, one with 70%
zeros, one near the smallest and one near the largest scale of binary64; the
element count leaves the last CTA of several one-warp blocks part empty.
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


def _blocks(E, n, seed):
    rng = np.random.default_rng(seed)
    D = rng.standard_normal((E, n, n))
    D[0] = np.round(2.0 * D[0]) / 2.0 + 7.0 * np.eye(n)
    D[1] *= 10.0 ** rng.integers(-12, 12, (n, 1)) * 10.0 ** rng.integers(-12, 12, (1, n))
    D[2] = D[2] * (rng.random((n, n)) < 0.3) + np.eye(n)
    D[3] *= 1e-300
    D[4] *= 1e300
    return D


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("dim,P", [(2, 0), (2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (3, 0), (3, 1), (3, 2), (3, 3)])
def test_register_factor_is_bit_identical_to_column_by_column(monkeypatch, dim, P, prec):
    from paper_1908_03972_gb300 import pmgfr
    nodes, nbr = W.periodic_box(3, 3, Ng=1) if dim == 2 else W.periodic_box3d(3, 3, 1, Ng=1)
    E, N = 9, (P + 1) ** dim
    n = (dim + 2) * N
    D = _blocks(E, n, 10 * n + prec)
    r = np.random.default_rng(3).standard_normal((dim + 2, E, N))
    out = []
    for force in (0, 8):
        monkeypatch.delenv("PMG_FACTOR_CLUSTER", raising=False)
        if force:
            monkeypatch.setenv("PMG_FACTOR_CLUSTER", str(force))
        s = pmgfr.Solver(nodes, nbr, [P], [1], block_prec=prec, dim=dim)
        try:
            pmgfr.pmg_set_blocks(s.h, 0, D)
            pmgfr.pmg_factor_blocks(s.h, 0)
            out.append(s.apply(r))
        finally:
            s.close()
    # FP32 scales of 1e300 overflow: those entries are NaN on both sides
    assert np.array_equal(out[0], out[1], equal_nan=True)
    assert np.isfinite(out[0][:, [0, 1, 2, 5, 6, 7, 8]]).all()

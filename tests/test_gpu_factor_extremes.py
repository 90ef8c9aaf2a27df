"""Factorisation of blocks whose rows reach the top of the binary64 range
(k_factor.cu): the power-of-two row scales are then subnormal, 2^-1023 and
2^-1024.

Rows multiplied by powers of two give the same equilibrated block, so with the
right-hand side multiplied alike the applied inverse is that of the block as it
was, bit for bit.  Where a column's entries leave the normal range under the row
scale (the column scales then come from the products themselves) the result is
that of the column-by-column kernel (PMG_FACTOR_CLUSTER = 8), bit for bit.  FP64
blocks only: FP32 and BF16 ones are applied to a right-hand side in FP32, which
does not reach these scales.
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


def _apply(dim, P, D, r):
    from paper_1908_03972_gb300 import pmgfr
    nodes, nbr = W.periodic_box(3, 3, Ng=1) if dim == 2 else W.periodic_box3d(3, 3, 1, Ng=1)
    s = pmgfr.Solver(nodes, nbr, [P], [1], block_prec=pmgfr.PMG_PREC_FP64, dim=dim)
    try:
        pmgfr.pmg_set_blocks(s.h, 0, D)
        pmgfr.pmg_factor_blocks(s.h, 0)
        return s.apply(r)
    finally:
        s.close()


SIZES = [(2, 0), (2, 1), (2, 2), (2, 3), (2, 4), (3, 0), (3, 1), (3, 2), (3, 3)]


def _base(dim, P):
    E, N = 9, (P + 1) ** dim
    n = (dim + 2) * N
    rng = np.random.default_rng(100 * n)
    B = rng.standard_normal((E, n, n)) + 2.0 * n ** 0.5 * np.eye(n)
    r = rng.standard_normal((dim + 2, E, N))
    ex = np.frexp(np.abs(B).max(axis=2))[1]                       # row maxima in [2^(ex-1), 2^ex)
    top = np.where(np.arange(n) % 3 == 0, 0, np.where(np.arange(n) % 3 == 1, 1023, 1024)) - ex
    return E, N, n, B, r, np.where(top < 0, 0, top)


@pytest.mark.parametrize("dim,P", SIZES)
def test_rows_near_the_largest_number(monkeypatch, dim, P):
    monkeypatch.delenv("PMG_FACTOR_CLUSTER", raising=False)
    E, N, n, B, r, s = _base(dim, P)
    r = r * 2.0 ** -8
    D = np.ldexp(B, s[:, :, None])
    assert np.isfinite(D).all() and (np.abs(D).max(axis=2) >= 2.0 ** 1022).any()
    rs = np.ldexp(r, np.moveaxis(s.reshape(E, dim + 2, N), 1, 0))
    plain, scaled = _apply(dim, P, B, r), _apply(dim, P, D, rs)
    assert np.isfinite(plain).all() and (plain != 0).any()
    assert np.array_equal(plain, scaled)


@pytest.mark.parametrize("dim,P", SIZES)
def test_columns_that_leave_the_normal_range(monkeypatch, dim, P):
    E, N, n, B, r, s = _base(dim, P)
    s = 1024 - np.frexp(np.abs(B).max(axis=2))[1]                 # every row scaled by 2^-1024
    D = np.ldexp(B, s[:, :, None])
    D[:, :, n // 2] = B[:, :, n // 2] / np.abs(B[:, :, n // 2]).max(axis=1, keepdims=True)   # below 2^-1022 then
    rs = np.ldexp(r * 2.0 ** -8, np.moveaxis(s.reshape(E, dim + 2, N), 1, 0))
    out = []
    for force in (None, "8"):
        monkeypatch.delenv("PMG_FACTOR_CLUSTER", raising=False)
        if force:
            monkeypatch.setenv("PMG_FACTOR_CLUSTER", force)
        out.append(_apply(dim, P, D, rs))
    assert np.isfinite(out[1]).all()
    assert np.array_equal(out[0], out[1])

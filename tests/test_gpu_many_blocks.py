"""Rules that depend on the number of blocks give the same numbers on both sides:
the first elements of a mesh with many blocks (the factorisation's layout for
many small FP64 blocks, k_factor.cu; the block apply's ring of asynchronous
copies for inverses beyond 80 MB, k3_blocks.cu, whose chunks start off 16-byte
boundaries at n = 135 and end with the array) against the same blocks on a mesh
of a few.  The operations on every entry are the same, in the same order, so the
results are equal.
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


@pytest.mark.parametrize("P,prec,many", [(2, 0, (28, 22)), (1, 0, (6, 6, 17)), (1, 0, (20, 20, 19)),
                                         (2, 0, (11, 10, 6)), (2, 1, (11, 11, 11)), (2, 2, (14, 14, 14)),
                                         (3, 0, (5, 5, 5)), (3, 1, (6, 7, 6)), (3, 2, (8, 8, 8))])
def test_same_blocks_in_small_and_large_numbers(P, prec, many):
    import torch
    from paper_1908_03972_gb300 import pmgfr
    dim = len(many)
    box = W.periodic_box if dim == 2 else W.periodic_box3d
    n = (dim + 2) * (P + 1) ** dim
    E = 1
    for k in many:
        E *= k
    few = (4, 4) if dim == 2 else (3, 2, 3)
    e = 16 if dim == 2 else 18
    g = torch.Generator(device="cuda").manual_seed(n + prec)
    D = torch.randn(E, n, n, device="cuda", dtype=torch.float64, generator=g)
    D += 0.5 * n ** 0.5 * torch.eye(n, device="cuda", dtype=torch.float64)
    r = torch.randn(dim + 2, E, n // (dim + 2), device="cuda", dtype=torch.float64, generator=g)
    out = []
    for size, which in ((many, slice(0, E)), (few, slice(0, e)), (few, slice(E - e, E))):
        s = pmgfr.Solver(*box(*size, Ng=1), [P], [1], block_prec=prec, dim=dim)
        try:
            Dk, rk = D[which].contiguous(), r[:, which].contiguous()
            x = torch.full_like(rk, float("nan"))
            torch.cuda.synchronize()
            pmgfr.pmg_set_blocks(s.h, 0, Dk)
            pmgfr.pmg_factor_blocks(s.h, 0)
            pmgfr.pmg_apply_blocks(s.h, 0, rk, x)
            torch.cuda.synchronize()
            out.append(x)
        finally:
            s.close()
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0][:, :e], out[1])
    assert torch.equal(out[0][:, E - e:], out[2])

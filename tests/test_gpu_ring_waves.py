"""The block apply on hexahedra (k3_blocks.cu) through its ring of asynchronous
copies where the ring's CTAs need more than one wave (n = 40 in FP32 and BF16, n =
135 in BF16, n = 320 in FP32) against the same blocks on a mesh of a few elements,
whose inverses go through registers: the same operations in the same order, so
the first and the last elements' results are equal.
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


@pytest.mark.parametrize("P,prec,many", [(1, 1, (24, 24, 23)), (1, 2, (30, 30, 29)), (2, 2, (19, 19, 23)),
                                         (3, 1, (17, 15, 10))])
def test_ring_in_several_waves(P, prec, many):
    import torch
    from paper_1908_03972_gb300 import pmgfr
    n, E, e = 5 * (P + 1) ** 3, many[0] * many[1] * many[2], 18
    g = torch.Generator(device="cuda").manual_seed(n + prec)
    D = torch.randn(E, n, n, device="cuda", dtype=torch.float64, generator=g)
    D += 0.5 * n ** 0.5 * torch.eye(n, device="cuda", dtype=torch.float64)
    r = torch.randn(5, E, n // 5, device="cuda", dtype=torch.float64, generator=g)
    out = []
    for size, which in ((many, slice(0, E)), ((3, 2, 3), slice(0, e)), ((3, 2, 3), slice(E - e, E))):
        s = pmgfr.Solver(*W.periodic_box3d(*size, Ng=1), [P], [1], block_prec=prec, dim=3)
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

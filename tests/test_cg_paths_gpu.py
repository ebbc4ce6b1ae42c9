"""The kernel paths of the CG iteration: the p update and <q,p> inside the apply or in kernels of their own, the
shared-node sums gathered in the preconditioner or in passes.  The size decides; every path has to
reach the residual it reports, recomputed with the FP64-pipe operator."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# one cell across an axis (no interface there), ragged boxes, and sizes on both sides of 400,000 and
# 1,048,576 entries (gathered sums in FP64 and FP32), of 4,194,304 (fused FP32 apply) and of 16 warps
# per SM (fused FP64 apply)
CASES = [(1, (2, 9, 8)), (2, (1, 9, 8)), (2, (7, 1, 5)), (3, (5, 6, 1)), (4, (1, 1, 7)), (7, (2, 1, 3)), (5, (4, 3, 5)),
         (2, (23, 25, 24)), (2, (25, 26, 27)), (3, (25, 25, 25)), (3, (25, 26, 27)), (6, (15, 13, 14)),
         (7, (12, 13, 14)), (7, (20, 20, 20)), (7, (21, 20, 20))]


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("p,m", CASES)
def test_reported_residual(p, m, mixed):
    from paper_2607_02335_gb300 import fe
    gm = fe.Mesh(m, p, deform_amp=0.1, dirichlet=True)
    g = torch.Generator(device="cuda").manual_seed(p)
    b = torch.rand(gm.cellwise_len, generator=g, device="cuda", dtype=torch.float64) - 0.5
    x = torch.zeros_like(b)
    res = gm.cg_solve(b, x, rtol=1e-10, maxit=4000, mixed=fe.FE_F32 if mixed else 0, inner_rtol=0.1)
    assert res.status == fe.FE_OK
    sb = gm.dss(b)
    ax = gm.apply(x, flags=fe.FE_ASSEMBLE | fe.FE_NATIVE_F64)
    ones = torch.ones_like(b)
    mult = gm.dss(ones)
    free = gm.apply(ones, op=fe.FE_MASS, flags=fe.FE_ASSEMBLE) != 0  # 0 on the Dirichlet nodes
    r = torch.where(free, sb - ax, 0.0)
    rel = ((r * r / mult).sum() / (torch.where(free, sb, 0.0) ** 2 / mult).sum()).sqrt().item()
    # the recursive residual and a recomputed one differ by rounding of the operator (1e-13 of |A||x|)
    assert rel <= 1.05e-10 + 1e-12, rel
    again = torch.zeros_like(b)
    gm.cg_solve(b, again, rtol=1e-10, maxit=4000, mixed=fe.FE_F32 if mixed else 0, inner_rtol=0.1)
    assert torch.equal(x, again)

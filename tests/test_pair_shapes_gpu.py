"""The tile shapes of the FP64 apply (single cells, small and ordinary tiles of cell pairs): the launch
size decides between them, and each against the FP64-pipe kernel, with a last pair that holds one cell
and a ragged last tile."""
import numpy as np
import pytest

from tests.helpers import rel_max_err

pytestmark = pytest.mark.gpu


def to_host(t):
    return t.cpu().numpy()


def box(cells):
    """An odd box of about `cells` cells."""
    m = max(1, round(cells ** (1 / 3)))
    m -= 1 - m % 2
    mz = max(1, round(cells / (m * m)))
    return (m, m, mz - 1 + mz % 2)


# cells x n^2 relative to the 512 threads per SM up to which single cells are taken
@pytest.mark.parametrize("share", [0.02, 0.9, 1.2, 2.3, 6.0])
@pytest.mark.parametrize("p", range(1, 8))
def test_shapes_equal_native(p, share):
    import torch
    from paper_2607_02335_gb300 import fe
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = box(max(1, int(share * 512 * sms / (p + 1) ** 2)))
    assert m[0] * m[1] * m[2] % 2 == 1
    for geom, amp in ((fe.FE_GEOM_STORED, 0.1), (fe.FE_GEOM_AFFINE, 0.0)):
        gm = fe.Mesh(m, p, deform_amp=amp, geom_mode=geom, dirichlet=geom == fe.FE_GEOM_STORED)
        g = torch.Generator(device="cuda").manual_seed(p)
        x = torch.rand(gm.cellwise_len, generator=g, device="cuda", dtype=torch.float64) - 0.5
        for op in (fe.FE_LAPLACE, fe.FE_MASS):
            y = torch.full((gm.cellwise_len + 2,), 7.0, device="cuda", dtype=torch.float64)
            gm.apply(x, op=op, y=y)
            ref = gm.apply(x, op=op, flags=fe.FE_NATIVE_F64)
            err = float((y[:-2] - ref).abs().max() / ref.abs().max())
            assert err <= 1e-12, (m, op, geom)  # the double-word path's bar against FP64
            assert y[-2:].tolist() == [7.0, 7.0]


# single cells; pairs (warp-wide and CTA-wide tiles)
@pytest.mark.parametrize("p,m", [(3, (3, 3, 3)), (3, (25, 25, 25)), (4, (21, 21, 21)), (7, (15, 13, 11))])
def test_nonfinite_stays_in_its_cell(p, m):
    import torch
    from paper_2607_02335_gb300 import fe
    n3 = (p + 1) ** 3
    gm = fe.Mesh(m, p, deform_amp=0.1)
    x = torch.rand(gm.cellwise_len, device="cuda", dtype=torch.float64) - 0.5
    for op in (fe.FE_LAPLACE, fe.FE_MASS):
        clean = to_host(gm.apply(x, op=op)).reshape(-1, n3)
        bad = x.clone()
        cells = {1: float("inf"), 6: float("nan"), gm.n_cells - 1: -float("inf")}
        for c, v in cells.items():
            bad[c * n3 + 2] = v
        y = to_host(gm.apply(bad, op=op)).reshape(-1, n3)
        for c in cells:
            assert not np.isfinite(y[c]).any(), (op, c)
        keep = np.ones(len(y), dtype=bool)
        keep[list(cells)] = False
        assert rel_max_err(y[keep], clean[keep]) <= 1e-14, op


def in_one_binade(gm, seed):
    """Random values of either sign with |x| in [1/2, 1): which cells hold them does not change the
    largest exponent of a tile."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(gm.cellwise_len, generator=g, device="cuda", dtype=torch.float64) - 0.5
    return torch.where(x < 0, x - 0.5, x + 0.5).clamp(-0.999, 0.999)


# single cells, warp-wide and CTA-wide tiles of pairs, with and without a small tile
@pytest.mark.parametrize("p,m", [(1, (9, 9, 9)), (1, (45, 45, 45)), (2, (13, 13, 13)), (3, (3, 3, 3)),
                                 (3, (25, 25, 25)), (4, (21, 21, 21)), (5, (17, 17, 17)), (6, (15, 15, 15)),
                                 (7, (5, 5, 5)), (7, (15, 13, 11))])
def test_bits_do_not_depend_on_the_tile(p, m):
    """A cell whose tile also holds an infinity or a NaN gets the bits it gets otherwise, and so does a mesh
    whose values lie outside the exponents of ordinary data (a power of two, exact in every step)."""
    import torch
    from paper_2607_02335_gb300 import fe
    n3 = (p + 1) ** 3
    gm = fe.Mesh(m, p, deform_amp=0.1)
    x = in_one_binade(gm, p)
    bad = x.clone()
    cells = {1: float("inf"), 6: float("nan"), gm.n_cells // 2: -float("inf"), gm.n_cells - 1: float("nan")}
    for c, v in cells.items():
        bad[c * n3 + 2] = v
    keep = torch.ones(gm.n_cells, dtype=torch.bool)
    keep[list(cells)] = False
    keep = keep.cuda()
    for op in (fe.FE_LAPLACE, fe.FE_MASS):
        clean = gm.apply(x, op=op)
        y = gm.apply(bad, op=op)
        assert torch.equal(y.view(-1, n3)[keep], clean.view(-1, n3)[keep]), op
        assert not y.view(-1, n3)[~keep].isfinite().any(), op
        for e in (900, -900):
            assert torch.equal(gm.apply(x * 2.0 ** e, op=op), clean * 2.0 ** e), (op, e)


@pytest.mark.parametrize("p,cells", [(1, 4), (2, 3), (3, 2), (3, 12), (4, 3), (5, 2), (6, 10), (7, 2)])
def test_overflow_of_the_metric_is_not_hidden(p, cells):
    """Blocks of side 1e16: w detJ is beyond the range of float, so the double-word mass apply of finite
    values overflows.  Its results are non-finite (or, were the range to grow, right), never other numbers."""
    import torch
    from paper_2607_02335_gb300 import fe, synth
    v, b, d = synth.mb_cube_in_cube(cells, seed=p)
    gm = fe.MBMesh(np.asarray(v) * 1e16, b, d, p)
    g = torch.Generator(device="cuda").manual_seed(p)
    x = torch.rand(gm.cellwise_len, generator=g, device="cuda", dtype=torch.float64) - 0.5
    y = gm.apply(x, op=fe.FE_MASS)
    ref = gm.apply(x, op=fe.FE_MASS, flags=fe.FE_NATIVE_F64)
    assert ref.isfinite().all() and ref.abs().max() > 1e36
    wrong = y.isfinite() & ((y - ref).abs() > 1e-12 * ref.abs().max())
    assert not wrong.any(), (int(wrong.sum()), y[wrong][:3].tolist(), ref[wrong][:3].tolist())

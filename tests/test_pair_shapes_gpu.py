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

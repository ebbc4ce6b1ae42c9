"""Recomputed geometry (metric formed on the fly from cell-wise nodal coordinates, Sec. 2.3 and
Sec. 6.2) against the FP64 CPU oracle and against the stored-metric mode of the same mesh.

The two modes describe the same operator, so they must agree to the FP64 bar (1e-12 relative
max-norm).  Meshes whose metric is larger than the scratch make the apply walk several chunks of cells
with a ragged last one."""
import os
import re

import numpy as np
import pytest

import oracle as O
from paper_2607_02335_gb300 import synth as S
from tests.helpers import oracle_mesh, rel_max_err, sampled_assembled

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL64 = 1e-12
TOL32 = 2e-5

SHAPES = {1: (5, 5, 5), 2: (5, 4, 3), 3: (5, 4, 3), 4: (7, 3, 3), 5: (5, 4, 3), 6: (7, 3, 3),
          7: (3, 3, 2)}


@pytest.fixture(scope="module")
def fe():
    from paper_2607_02335_gb300 import fe as F
    return F


def to_host(t):
    return t.detach().cpu().numpy().astype(np.float64)


def scratch_bytes(name):
    """A scratch size of the library's source."""
    src = open(os.path.join(os.path.dirname(os.path.abspath(__file__)), os.pardir, "paper_2607_02335_gb300",
                            "csrc", "fe_internal.h")).read()
    return int(re.search(rf"#define {name} \((\d+)LL << 20\)", src).group(1)) << 20


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
def test_recompute_vs_oracle_and_stored(fe, p):
    m = SHAPES[p]
    om = oracle_mesh(m, p, amp=0.1)
    gr = fe.Mesh(m, p, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE)
    gs = fe.Mesh(m, p, deform_amp=0.1, geom_mode=fe.FE_GEOM_STORED)
    xc = O.gather(om, S.primal_unique(m, p, seed=1))
    x = torch.from_numpy(xc).cuda()
    for op in (fe.FE_LAPLACE, fe.FE_MASS):
        yref = O.apply_local(om, op, xc)
        yr = to_host(gr.apply(x, op=op))
        assert rel_max_err(yr, yref) <= TOL64, (p, op)
        assert rel_max_err(yr, to_host(gs.apply(x, op=op))) <= TOL64, (p, op, "stored")
        yn = to_host(gr.apply(x, op=op, flags=fe.FE_NATIVE_F64))
        assert rel_max_err(yn, yref) <= TOL64, (p, op, "native")
        y32 = to_host(gr.apply(x.float(), op=op, prec=fe.FE_F32))
        assert rel_max_err(y32, yref) <= TOL32, (p, op, "fp32")


@pytest.mark.parametrize("p,m", [(2, (4, 3, 5)), (5, (2, 3, 2))])
def test_recompute_assembled_dirichlet_and_diag(fe, p, m):
    om = oracle_mesh(m, p, amp=0.1, dirichlet=True)
    gm = fe.Mesh(m, p, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE, dirichlet=True)
    xg = S.primal_unique(m, p, seed=3, dirichlet=True)
    x = gm.gather(xg)
    for op in (O.LAPLACE, O.MASS):
        yref = O.gather(om, O.apply_dirichlet_csr(om, O.assemble_csr(om, op), xg))
        y = to_host(gm.apply(x, op=op, flags=fe.FE_ASSEMBLE))
        assert rel_max_err(y, yref) <= TOL64, op
        dref = O.gather(om, O.diag_global(om, op))
        assert rel_max_err(to_host(gm.diag(op)), dref) <= TOL64, op


@pytest.mark.parametrize("p,m", [(3, 54), (7, (26, 27, 28)), (1, 108)])
def test_recompute_several_chunks(fe, p, m):
    """Sizes whose metric spans several scratch chunks (the last one ragged): recompute equals
    stored over the whole vector in every arithmetic, and sampled entries match the oracle."""
    gr = fe.Mesh(m, p, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE)
    assert 7 * 4 * gr.cellwise_len > scratch_bytes("FE_RC_CHUNK_BYTES")  # in FP32, the smaller one
    gs = fe.Mesh(m, p, deform_amp=0.1)
    xg = S.primal_unique(m, p, seed=2)
    x = gr.gather(xg)
    for op in (fe.FE_LAPLACE, fe.FE_MASS):
        yr = gr.apply(x, op=op, flags=fe.FE_ASSEMBLE)
        ys = gs.apply(x, op=op, flags=fe.FE_ASSEMBLE)
        scale = ys.abs().max().item()
        assert (yr - ys).abs().max().item() <= TOL64 * scale, op
        yr32 = gr.apply(x.float(), op=op, prec=fe.FE_F32)
        ys32 = gs.apply(x.float(), op=op, prec=fe.FE_F32)
        s32 = ys32.abs().max().item()
        assert (yr32 - ys32).abs().max().item() <= TOL32 * s32, op
        del yr32, ys32
        om = oracle_mesh(m, p, amp=0.1)
        rng = np.random.default_rng(p)
        n3 = (p + 1) ** 3
        samples = [(int(c), int(l)) for c, l in zip(rng.integers(0, gr.n_cells, 8),
                                                    rng.integers(0, n3, 8))]
        samples += [(gr.n_cells - 1, n3 - 1)]
        got = np.array([yr[c * n3 + l].item() for c, l in samples])
        ref = sampled_assembled(om, op, xg, samples)
        assert np.abs(got - ref).max() <= TOL64 * scale, op


@pytest.mark.parametrize("p,m", [(1, (65, 63, 67)), (2, (35, 35, 37)), (3, (25, 25, 27)),
                                 (4, (19, 19, 21)), (5, (15, 17, 17)), (6, (13, 13, 15)),
                                 (7, (13, 13, 15)), (3, (44, 45, 47))])
def test_recompute_pairs_and_ragged_chunks(fe, p, m):
    """Meshes large enough for the kernels on pairs of cells, with an odd number of cells (the last
    pair has one cell), and one whose metric spans two scratch chunks: recompute equals stored.  The
    bounds are those of the oracle comparisons above, which both sides meet."""
    gr = fe.Mesh(m, p, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE)
    gs = fe.Mesh(m, p, deform_amp=0.1)
    x = torch.from_numpy(S.dual_cellwise(m, p, seed=4)).cuda()
    for op in (fe.FE_LAPLACE, fe.FE_MASS):
        for kw, v, tol in (({}, x, TOL64), ({"prec": fe.FE_F32}, x.float(), TOL32)):
            ys = gs.apply(v, op=op, **kw)
            err = (gr.apply(v, op=op, **kw) - ys).abs().max().item()
            assert err <= tol * ys.abs().max().item(), (op, kw)
    gr.close()
    gs.close()


# odd and even n, more than 256 MB of FP32 metric, the last chunk ragged
@pytest.mark.parametrize("p,m", [(2, (71, 73, 71)), (3, (54, 55, 53)), (4, (43, 43, 45)), (5, (37, 35, 37))])
def test_recompute_several_chunks_in_every_arithmetic(fe, p, m):
    """Meshes whose metric spans several scratch chunks in FP64, on the FP64 pipe, in FP32 and for the
    diagonal: recompute equals stored, unassembled and assembled.  The bounds are those of the oracle
    comparisons above, which both sides meet."""
    gr = fe.Mesh(m, p, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE)
    gs = fe.Mesh(m, p, deform_amp=0.1)
    entries = gr.cellwise_len
    assert 7 * 4 * entries > scratch_bytes("FE_RC_CHUNK_BYTES")
    assert 7 * 8 * entries > scratch_bytes("FE_RC_DIAG_BYTES")
    g = torch.Generator(device="cuda").manual_seed(p)
    x = torch.rand(entries, generator=g, dtype=torch.float64, device="cuda") - 0.5
    for op in (fe.FE_LAPLACE, fe.FE_MASS):
        for kw, v, tol in (({}, x, TOL64), ({"flags": fe.FE_ASSEMBLE}, x, TOL64),
                           ({"flags": fe.FE_NATIVE_F64}, x, TOL64), ({"prec": fe.FE_F32}, x.float(), TOL32)):
            ys = gs.apply(v, op=op, **kw)
            err = (gr.apply(v, op=op, **kw) - ys).abs().max().item()
            assert err <= tol * ys.abs().max().item(), (op, kw)
        ds = gs.diag(op)
        assert (gr.diag(op) - ds).abs().max().item() <= TOL64 * ds.abs().max().item(), op
    gr.close()
    gs.close()


def test_recompute_cg_matches_stored(fe):
    """Jacobi-PCG on a recompute mesh takes the same path as on the stored mesh."""
    m, p = (5, 4, 3), 3
    bc = S.dual_cellwise(m, p, seed=21)
    out = {}
    for mode in (fe.FE_GEOM_STORED, fe.FE_GEOM_RECOMPUTE):
        gm = fe.Mesh(m, p, deform_amp=0.1, geom_mode=mode, dirichlet=True)
        x = torch.zeros(gm.cellwise_len, dtype=torch.float64, device="cuda")
        res, hist = gm.cg_solve(torch.from_numpy(bc).cuda(), x, rtol=1e-11, maxit=500,
                                history=True)
        assert res.status == fe.FE_OK
        out[mode] = (res, hist, to_host(x))
        xm = torch.zeros_like(x)
        rm = gm.cg_solve(torch.from_numpy(bc).cuda(), xm, rtol=1e-10, maxit=500,
                         mixed=fe.FE_F32, flexible=True)
        assert rm.status == fe.FE_OK and rm.rel_res <= 1e-10
    (rs, hs, xs), (rr, hr, xr) = out[fe.FE_GEOM_STORED], out[fe.FE_GEOM_RECOMPUTE]
    assert abs(rs.iters - rr.iters) <= 1
    k = min(rs.iters, rr.iters, 20)
    assert np.allclose(hs[:k, 0], hr[:k, 0], rtol=1e-9, atol=0)
    assert rel_max_err(xr, xs) <= 1e-9


def test_recompute_not_accepted_by_batched(fe):
    gm = fe.Mesh(2, 2, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE)
    b = torch.ones(gm.cellwise_len, dtype=torch.float64, device="cuda")
    x = torch.zeros_like(b)
    with pytest.raises(fe.FeError):
        fe.fe_cg_solve_batched([gm.handle], [b], [x], fe.fe_cg_opts(1e-8, 10, 0, 0, 1e-2, None))


def test_scratch_is_shared_between_arithmetics(fe):
    """What a recompute mesh holds on the device after applies in every arithmetic and a diagonal: the
    coordinate copies, one metric scratch of 256 MB (allocated with the mesh) and the diagonal's 48 MB."""
    gm = fe.Mesh((54, 54, 53), 3, deform_amp=0.1, geom_mode=fe.FE_GEOM_RECOMPUTE)
    n = gm.cellwise_len
    assert 7 * 4 * n > 256 << 20  # the metric is beyond the scratch in FP32 too
    x = torch.rand(n, dtype=torch.float64, device="cuda")
    y, x32, y32 = torch.empty_like(x), x.float(), torch.empty(n, dtype=torch.float32, device="cuda")
    gm.apply(x, y=y)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    gm.apply(x32, prec=fe.FE_F32, y=y32)
    gm.apply(x, flags=fe.FE_NATIVE_F64, y=y)
    fe.fe_diag(gm.handle, fe.FE_LAPLACE, y)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    coords32 = 3 * 4 * n
    # 128 MB: the device pool's growth in large steps, and the kernels loaded by their first launch
    assert used <= coords32 + (48 << 20) + (128 << 20), used / 2 ** 20
    gm.close()

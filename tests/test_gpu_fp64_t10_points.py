"""FP64 operations on affine T10 blocks (one CTA per tile, one warp per
quadrature point) at the sizes where their tiling can go wrong: one tile with
most of its lanes padding, one lane into a second tile, and more tiles than
the GPU holds CTAs (the double-buffered metadata and the gather of the next
tile), with both rules, a mass term, and the one-pass force + operator
product. Tolerance: the FP64 parity bar of the other tests, 1e-12 of the
largest value."""

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

H = 1e-3


def relerr(got, ref):
    return np.abs(got.cpu().numpy() - ref).max() / np.abs(ref).max()


# cells -> elements: 6 (one ragged tile), 36 (one tile and 4 lanes), 10,368 (324 tiles, two per CTA somewhere)
@pytest.mark.parametrize("cells,n_elem", [((1, 1, 1), 6), ((3, 2, 1), 36), ((12, 12, 12), 10368)])
@pytest.mark.parametrize("nq,scatter", [(4, 0), (5, 0), (5, 2)])
def test_matches_the_oracle(cells, n_elem, nq, scatter):
    from paper_2602_17002_gb300 import tlfe as tl
    wl = synth.cantilever_beam(cells=cells, nq=nq)
    assert wl.n_elem == n_elem
    mesh = tl.Mesh.from_workload(wl, precision=tl.FP64, scatter=scatter)
    assert mesh.info["force_matvec_fused"] == 1
    u, ud, v = (torch.from_numpy(a).cuda() for a in (wl.u, wl.udot, wl.v))
    f, y = mesh.force_matvec(u, ud, v, 1.0 / H, H, 1.0)
    f2, y2 = mesh.internal_force(u, ud), mesh.tangent_matvec(u, ud, v, 1.0 / H, H, 1.0)
    ym = mesh.tangent_matvec(u, None, v, 1.0 / H, 0.0, 0.0)          # the mass product alone
    gu, gud, gth = mesh.vjp(u, ud, v)
    assert mesh.sync() == 0
    f_ref, _ = oracle.internal_force(wl)
    y_ref = oracle.operator_apply(wl, wl.v, a_M=1.0 / H, a_K=H, a_C=1.0)
    gu_ref, gud_ref, gth_ref = oracle.vjp(wl, wl.v)
    for got, ref in ((f, f_ref), (f2, f_ref), (y, y_ref), (y2, y_ref), (gu, gu_ref), (gud, gud_ref), (gth, gth_ref),
                     (ym, oracle.operator_apply(wl, wl.v, a_M=1.0 / H, a_K=0.0, a_C=0.0, udot=None))):
        assert relerr(got, ref) <= 1e-12
    mesh.close()


def test_undamped_adjoint_has_a_zero_velocity_gradient():
    from paper_2602_17002_gb300 import tlfe as tl
    wl = synth.block_t10_svk(cells=2)
    mesh = tl.Mesh.from_workload(wl, precision=tl.FP64)
    u, v = torch.from_numpy(wl.u).cuda(), torch.from_numpy(wl.v).cuda()
    gu, gud, _ = mesh.vjp(u, None, v)
    mesh.sync()
    assert relerr(gu, oracle.vjp(wl, wl.v)[0]) <= 1e-12
    assert not gud.any()
    mesh.close()

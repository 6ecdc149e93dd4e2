"""FP32 operations on affine T10 and H8 blocks, whose points are evaluated two
at a time from the lane's own shared-memory column, at the sizes where their
tiling can go wrong (a ragged tile, a few lanes into a second tile, more tiles
than resident warps), for both T10 rules, every law with and without damping,
with and without a mass term, and with points of one pair on both sides of
J = 0. Tolerance: the FP32 parity bar of the other tests, 2e-5 of the largest
value."""

import numpy as np
import pytest

import oracle
import synth
from synth.mesh import box_mesh
from synth.workloads import Block, Workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-5
H = 1e-3


def T():
    from paper_2602_17002_gb300 import tlfe
    return tlfe


def relerr(got, ref):
    return np.abs(got.double().cpu().numpy() - ref).max() / np.abs(ref).max()


def _box(etype, nq, cells, law, damped, seed=3):
    m = box_mesh(etype, cells, tuple(0.05 * c for c in cells))
    rng = np.random.default_rng(seed)
    shape = m.X.shape
    S = rng.uniform(-0.05, 0.05, (3, 3))
    u = m.X @ S + rng.uniform(-5e-4, 5e-4, shape)
    params = [3.8e6, 5.8e6, 1e3 if damped else 0.0, 2e2 if damped else 0.0, 1000.0] + ([5e5] if law == 2 else [])
    return Workload("box", m.X, [Block(etype, nq, m.conn, m.body)], np.array([law], np.int32), np.array([params]), u=u,
                    udot=0.01 * rng.standard_normal(shape), v=rng.standard_normal(shape))


def _run(wl, scatter, mass):
    tl = T()
    mesh = tl.Mesh.from_workload(wl, precision=tl.FP32, scatter=scatter)
    assert mesh.info["n_affine_blocks"] == 1
    u = torch.from_numpy(wl.u).cuda()
    ud, v = (torch.from_numpy(a).cuda().float() for a in (wl.udot, wl.v))
    a = (1.0 / H, H, 1.0) if mass else (0.0, 1.0, 1.0)
    f, y = mesh.force_matvec(u, ud, v, *a)
    out = [f, y, mesh.internal_force(u, ud), mesh.tangent_matvec(u, ud, v, *a), *mesh.vjp(u, ud, v)]
    assert mesh.sync() == 0
    mesh.close()
    f_ref, _ = oracle.internal_force(wl)
    y_ref = oracle.operator_apply(wl, wl.v, a_M=a[0], a_K=a[1], a_C=a[2])
    gu, gud, gth = oracle.vjp(wl, wl.v)
    for got, ref in zip(out, (f_ref, y_ref, f_ref, y_ref, gu, gud, gth)):
        if np.abs(ref).max() > 0:
            assert relerr(got, ref) <= TOL
        else:
            assert not got.any()


@pytest.mark.parametrize("etype,nq", [(synth.T10, 4), (synth.T10, 5), (synth.H8, 8)])
@pytest.mark.parametrize("law,damped", [(0, False), (0, True), (1, False), (1, True), (2, True)])
def test_laws_match_the_oracle(etype, nq, law, damped):
    _run(_box(etype, nq, (3, 2, 2), law, damped), 0, mass=law != 2)


# cells of one T10 tile with padding, a second tile of few lanes, and more tiles than warps fit an SM's share
@pytest.mark.parametrize("etype,nq,cells", [(synth.T10, 5, (1, 1, 1)), (synth.T10, 5, (3, 2, 1)), (synth.H8, 8, (1, 1, 1)),
                                            (synth.H8, 8, (11, 3, 1)), (synth.T10, 4, (24, 22, 21)),
                                            (synth.H8, 8, (41, 40, 41))])
@pytest.mark.parametrize("scatter", [0, 2])
def test_tile_edges_match_the_oracle(etype, nq, cells, scatter):
    _run(_box(etype, nq, cells, 1, cells[0] < 20), scatter, mass=cells[0] < 20)


@pytest.mark.parametrize("etype,nq", [(synth.T10, 4), (synth.T10, 5), (synth.H8, 8)])
def test_inverted_points_beside_good_ones(etype, nq):
    """One node moved by three cell edges turns some points of its elements
    inside out: they are counted, drop their elastic part, and leave the other
    point of their pair alone, as the FP64 kernels (other code) do."""
    tl = T()
    wl = _box(etype, nq, (2, 2, 2), 1, True)
    wl.u[wl.blocks[0].conn[5, 0]] += 0.15
    out = {}
    for prec in (tl.FP64, tl.FP32):
        mesh = tl.Mesh.from_workload(wl, precision=prec)
        u = torch.from_numpy(wl.u).cuda()
        ud, v = (torch.from_numpy(a).cuda().to(mesh.torch_dtype) for a in (wl.udot, wl.v))
        f = mesh.internal_force(u, ud)
        with pytest.raises(tl.TLFEError) as e:
            mesh.sync()
        out[prec] = (str(e.value), f, mesh.tangent_matvec(u, ud, v, 0.0, 1.0, 1.0), *mesh.vjp(u, ud, v))
        with pytest.raises(tl.TLFEError):
            mesh.sync()
        mesh.close()
    assert out[tl.FP64][0] == out[tl.FP32][0] and "J <= 0" in out[tl.FP32][0]      # the same number of points
    for a, b in zip(out[tl.FP32][1:], out[tl.FP64][1:]):
        assert relerr(a, b.cpu().numpy()) <= TOL

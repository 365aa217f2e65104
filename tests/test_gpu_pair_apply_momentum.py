"""The FP32 momentum apply of the persistent kernel (CHNS_APPLY_STREAM; a thread's two leaves one after
the other, pairs of Gauss points in packed arithmetic): meshes of one leaf, a lone brick, odd
numbers of leaves outside bricks and many hanging slots, a stretched box, FP32 and bfloat16
coefficients, one CTA for all patches; against the oracle's matrix on the same rounded inputs and
against the CTA-per-patch kernel; and its form on quadrature data inside a solve.

Bounds: 1e-5 against the oracle as for the other FP32 applies; the two kernels differ in the order
of their sums, in chains of about 40 roundings of 6e-8 that mostly agree: 4e-6."""
import numpy as np
import pytest

from gpu_common import PRM, bf16_round, dev, f32_round, fields, meshes, oracle_operator, relerr
from test_gpu_pair_apply import MESHES

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402
from oracle.mesh import Mesh as OMesh  # noqa: E402


def _coef(phi, u, mu, dtype=torch.float32, one=0.0):
    return capi.make_coef(dev(phi + one, dtype), [dev(v, dtype) for v in u], dev(mu, dtype))


def _run(gm, coef, x, prec, kernel):
    capi.chns_mesh_set_apply_config(gm.handle, kernel, 1 if kernel == capi.APPLY_STREAM else 0)
    y = torch.full((x.numel(),), 7.0, dtype=torch.float32, device="cuda")
    capi.chns_apply_momentum(gm.handle, capi.make_params(PRM), coef, x, y, prec)
    return y.double().cpu().numpy()


@pytest.mark.parametrize("prec", [capi.FP32, capi.FP32_BF16COEF])
@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("extent", [(1.0, 1.0, 1.0), (1.0, 2.0, 0.5)])
def test_pair_apply_momentum(name, extent, prec):
    a, l = MESHES[name]()
    om, gm = OMesh(a, l, extent), Mesh(a, l, extent)
    f = fields(om.n_nodes, 31)
    x = f32_round(f["x"].ravel())
    if prec == capi.FP32:
        phi, u, mu = f32_round(f["phi"]), f32_round(f["u"]), f32_round(f["mu"])
        coef = _coef(phi, u, mu)
    else:
        phi, u, mu = bf16_round(1.0 + f["phi"]) - 1.0, bf16_round(f["u"]), bf16_round(f["mu"])
        coef = _coef(phi, u, mu, torch.bfloat16, 1.0)
    ref = oracle_operator(om, capi.OP_MOMENTUM, PRM, phi, u, mu) @ x
    xd = dev(x, torch.float32)
    y = _run(gm, coef, xd, prec, capi.APPLY_STREAM)
    assert relerr(y, ref) < 1e-5
    assert relerr(y, _run(gm, coef, xd, prec, capi.APPLY_PATCH)) < 4e-6
    gm.close()


def test_pair_apply_momentum_keeps_nan_where_it_belongs():
    """A NaN of x reaches the nodes the CTA-per-patch kernel takes it to and no others."""
    gm = Mesh(*MESHES["random_l2_5"]())
    f = fields(gm.n_nodes, 3)
    x = f["x"].copy()
    x[1][np.flatnonzero(~gm.boundary)[7]] = np.nan
    coef, xd = _coef(f["phi"], f["u"], f["mu"]), dev(x.ravel(), torch.float32)
    y = _run(gm, coef, xd, capi.FP32, capi.APPLY_STREAM)
    assert np.isnan(y).any()
    assert np.array_equal(np.isnan(y), np.isnan(_run(gm, coef, xd, capi.FP32, capi.APPLY_PATCH)))
    gm.close()


@pytest.mark.parametrize("kernel", [capi.APPLY_PATCH, capi.APPLY_STREAM])
@pytest.mark.parametrize("name", ["one_refined", "random0_box", "random1", "drop_l3_5"])
def test_momentum_solve_on_quadrature_data(name, kernel):
    """FP32 GMRES refined in FP64 reaches the FP64 residual the oracle's matrix confirms (5 % for
    the rounding of the residual itself, as in the other mixed-precision solves)."""
    om, gm = meshes(name)
    f = fields(om.n_nodes, 41)
    A = oracle_operator(om, capi.OP_MOMENTUM, PRM, f["phi"], f["u"], f["mu"])
    b = f["x"].ravel().copy()
    coef = capi.make_coef(dev(f["phi"]), [dev(v) for v in f["u"]], dev(f["mu"]))
    x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    capi.chns_mesh_set_apply_config(gm.handle, kernel, 0)
    try:
        st = capi.chns_krylov_solve(gm.handle, capi.OP_MOMENTUM, capi.make_params(PRM), coef, dev(b),
                                    x, capi.make_solver(capi.KSP_GMRES, capi.PC_JACOBI, 1e-10, 4000,
                                                        30, capi.FP32, 1e-4))
    finally:
        capi.chns_mesh_set_apply_config(gm.handle, capi.APPLY_AUTO, 0)
    assert st.status == capi.OK and st.refinements >= 1
    assert np.linalg.norm(b - A @ x.cpu().numpy()) / np.linalg.norm(b) <= 1.05e-10

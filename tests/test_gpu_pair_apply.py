"""The FP32 applies with two leaves per thread (CHNS_APPLY_STREAM) where they can go wrong: a mesh of
one leaf, a lone brick, odd numbers of leaves outside bricks, patches with many hanging slots, more
slots than are loaded ahead, FP32 and bfloat16 coefficients, one CTA for all patches; against the
oracle's matrix on the same rounded inputs and against the CTA-per-patch kernel.

Bounds: an element result is a chain of about 20 roundings of 6e-8, sums of up to about 30 terms,
so 1e-5 against the oracle (as for the other FP32 applies) and 2e-6 between the kernels."""
import numpy as np
import pytest

from chns_workloads import configs, octree
from gpu_common import LEAVES, PRM, bf16_round, dev, f32_round, fields, oracle_operator, relerr

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402
from oracle.mesh import Mesh as OMesh  # noqa: E402

APPLY = {capi.OP_POISSON: capi.chns_apply_poisson, capi.OP_MASS: capi.chns_apply_mass}
MESHES = {
    "root": lambda: octree.uniform(0),
    "brick": lambda: octree.uniform(1),
    "uniform3": lambda: octree.uniform(3),
    "one_refined": LEAVES["one_refined"][0],
    "random_l1_6": lambda: configs.random_balanced(9, 1, 6, 0.3),
    "random_l2_5": lambda: configs.random_balanced(1, 2, 5, 0.2),
}


def _run(gm, op, coef, x, prec, kernel):
    capi.chns_mesh_set_apply_config(gm.handle, kernel, 1 if kernel == capi.APPLY_STREAM else 0)
    y = torch.full((x.numel(),), 7.0, dtype=torch.float32, device="cuda")
    APPLY[op](gm.handle, capi.make_params(PRM), coef, x, y, prec)
    return y.double().cpu().numpy()


@pytest.mark.parametrize("prec", [capi.FP32, capi.FP32_BF16COEF])
@pytest.mark.parametrize("op", [capi.OP_POISSON, capi.OP_MASS])
@pytest.mark.parametrize("name", list(MESHES))
def test_pair_apply(name, op, prec):
    a, l = MESHES[name]()
    om, gm = OMesh(a, l), Mesh(a, l)
    f = fields(om.n_nodes, 5 + op)
    x = f32_round(f["x"][:capi.OP_NCOMP[op]].ravel())
    if prec == capi.FP32:
        phi = f32_round(f["phi"])
        coef = capi.make_coef(dev(phi, torch.float32))
    else:
        phi = bf16_round(1.0 + f["phi"]) - 1.0
        coef = capi.make_coef(dev(1.0 + phi, torch.bfloat16))
    ref = oracle_operator(om, op, PRM, phi) @ x
    xd = dev(x, torch.float32)
    y = _run(gm, op, coef, xd, prec, capi.APPLY_STREAM)
    assert relerr(y, ref) < 1e-5
    assert relerr(y, _run(gm, op, coef, xd, prec, capi.APPLY_PATCH)) < 2e-6
    gm.close()


@pytest.mark.parametrize("op", [capi.OP_POISSON, capi.OP_MASS])
def test_pair_apply_keeps_nan_where_it_belongs(op):
    """A NaN of phi or x reaches the nodes of the leaves it is in and no others."""
    a, l = MESHES["random_l2_5"]()
    gm = Mesh(a, l)
    f = fields(gm.n_nodes, 3)
    for which in ("phi", "x"):
        phi, x = f["phi"].copy(), f["x"][:capi.OP_NCOMP[op]].copy()
        inner = np.flatnonzero(~gm.boundary)[7]
        (phi if which == "phi" else x[0])[inner] = np.nan
        coef, xd = capi.make_coef(dev(phi, torch.float32)), dev(x.ravel(), torch.float32)
        y = _run(gm, op, coef, xd, capi.FP32, capi.APPLY_STREAM)
        yp = _run(gm, op, coef, xd, capi.FP32, capi.APPLY_PATCH)
        assert np.isnan(y).any()
        assert np.array_equal(np.isnan(y), np.isnan(yp))
    gm.close()

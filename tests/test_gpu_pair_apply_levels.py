"""The FP32 applies on octrees refined towards a corner through every level up to 16, 17 and 19: chains
of leaves of which one patch's worth spans more levels than a reference of the two-leaves-per-thread
kernel can tell apart (patches are closed before). All four operators, FP32 and bfloat16
coefficients, both kernels and the automatic choice, against the oracle's matrix on the same rounded
inputs.

Bound: node by node, since a norm over all nodes sees the coarse ones only (the entries of the mass
matrix fall by 8 per level). Rounding of a row is bounded by 1e-5 (chains of about 40 roundings of
6e-8 and sums of up to 30 terms, as for the other FP32 applies) of the sum of its absolute
products."""
import numpy as np
import pytest

from chns_workloads import octree
from gpu_common import PRM, bf16_round, dev, f32_round, fields, oracle_operator

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402
from oracle.mesh import Mesh as OMesh  # noqa: E402

APPLY = {capi.OP_POISSON: capi.chns_apply_poisson, capi.OP_MASS: capi.chns_apply_mass,
         capi.OP_CH: capi.chns_apply_ch, capi.OP_MOMENTUM: capi.chns_apply_momentum}


def corner_octree(lmax, upper):
    at = (1 << octree.MAXD) if upper else 0

    def refine(x, level):
        return (x + (1 << (octree.MAXD - level)) * upper == at).all(axis=1)

    return octree.morton_sort(*octree.build_octree(refine, 1, lmax))


@pytest.mark.parametrize("prec", [capi.FP32, capi.FP32_BF16COEF])
@pytest.mark.parametrize("op", list(APPLY))
@pytest.mark.parametrize("upper", [0, 1])
@pytest.mark.parametrize("lmax", [16, 17, 19])
def test_pair_apply_levels(lmax, upper, op, prec):
    a, l = corner_octree(lmax, upper)
    assert l.max() == lmax and l.min() == 1
    om, gm = OMesh(a, l), Mesh(a, l)
    f = fields(om.n_nodes, 51 + op)
    x = f32_round(f["x"][:capi.OP_NCOMP[op]].ravel())
    if prec == capi.FP32:
        phi, u, mu = f32_round(f["phi"]), f32_round(f["u"]), f32_round(f["mu"])
        dt, one = torch.float32, 0.0
    else:
        phi, u, mu = bf16_round(1.0 + f["phi"]) - 1.0, bf16_round(f["u"]), bf16_round(f["mu"])
        dt, one = torch.bfloat16, 1.0
    coef = capi.make_coef(dev(phi + one, dt), [dev(v, dt) for v in u], dev(mu, dt))
    A = oracle_operator(om, op, PRM, phi, u, mu)
    ref, scale = A @ x, abs(A) @ np.abs(x)
    xd = dev(x, torch.float32)
    for kernel in (capi.APPLY_STREAM, capi.APPLY_PATCH, capi.APPLY_AUTO):
        capi.chns_mesh_set_apply_config(gm.handle, kernel, 0)
        y = torch.full((x.size,), 7.0, dtype=torch.float32, device="cuda")
        APPLY[op](gm.handle, capi.make_params(PRM), coef, xd, y, prec)
        err = np.abs(y.double().cpu().numpy() - ref) / scale
        assert err.max() < 1e-5, (kernel, err.max())
    gm.close()

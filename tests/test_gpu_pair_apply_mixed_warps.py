"""The FP32 Poisson, mass and shifted applies with two leaves per thread on meshes nearly every patch
of which has a warp with brick pairs and other leaves that share nodes: both kinds add to the same
sums, one after the other. Many runs, each against the oracle's matrix node by node (a lost
contribution is a large share of its node's sum, and may hide in a norm), and the shifted operator
through V-cycles of the multigrid hierarchy.

Bounds: 1e-5 of the sum of a row's absolute products (chains of about 40 roundings of 6e-8, sums of
up to 30 terms); 1e-4 for an FP32 V-cycle, as for the Poisson V-cycles."""
import numpy as np
import pytest

from chns_workloads import configs
from gpu_common import PRM, bf16_round, dev, f32_round, fields, oracle_operator, relerr
from oracle import multigrid as omg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402
from oracle.mesh import Mesh as OMesh  # noqa: E402

APPLY = {capi.OP_POISSON: capi.chns_apply_poisson, capi.OP_MASS: capi.chns_apply_mass}
MESHES = {"l1_6": (9, 1, 6, 0.3), "l2_6": (3, 2, 6, 0.15), "l3_6": (4, 3, 6, 0.1)}
RUNS = 50


@pytest.mark.parametrize("prec", [capi.FP32, capi.FP32_BF16COEF])
@pytest.mark.parametrize("op", list(APPLY))
@pytest.mark.parametrize("name", list(MESHES))
def test_mixed_warps(name, op, prec):
    a, l = configs.random_balanced(*MESHES[name])
    om, gm = OMesh(a, l), Mesh(a, l)
    f = fields(om.n_nodes, 61 + op)
    x = f32_round(f["x"][:capi.OP_NCOMP[op]].ravel())
    if prec == capi.FP32:
        phi = f32_round(f["phi"])
        coef = capi.make_coef(dev(phi, torch.float32))
    else:
        phi = bf16_round(1.0 + f["phi"]) - 1.0
        coef = capi.make_coef(dev(1.0 + phi, torch.bfloat16))
    A = oracle_operator(om, op, PRM, phi)
    ref, scale = A @ x, abs(A) @ np.abs(x)
    xd = dev(x, torch.float32)
    y = torch.empty(x.size, dtype=torch.float32, device="cuda")
    for run in range(RUNS):
        capi.chns_mesh_set_apply_config(gm.handle, capi.APPLY_STREAM, run % 3)
        APPLY[op](gm.handle, capi.make_params(PRM), coef, xd, y, prec)
        err = (np.abs(y.double().cpu().numpy() - ref) / scale).max()
        assert err < 1e-5, run
    gm.close()


@pytest.mark.parametrize("name", list(MESHES))
def test_mixed_warps_shifted(name):
    a, l = configs.random_balanced(*MESHES[name])
    om, gm = OMesh(a, l), Mesh(a, l)
    sa = 1.0 / np.sqrt(PRM["dt"])
    sb = PRM["Cn"] * np.sqrt(0.5 / (PRM["Pe"] * PRM["Cn"]))
    oms = omg.hierarchy(om.anchors, om.levels, om.extent, coarsest_level=2)
    r = f32_round(np.random.default_rng(14).standard_normal(om.n_nodes))
    ref = omg.VCycle(oms, PRM, shift=(sa, sb), degree=3)(r)
    mg = capi.chns_mg_create(gm.handle, coarsest_level=2, degree=3)
    try:
        for run in range(5):
            capi.chns_mesh_set_apply_config(gm.handle, capi.APPLY_STREAM, run % 3)
            capi.chns_mg_setup_shifted(mg, capi.make_params(PRM), sa, sb, capi.FP32)
            z = torch.zeros(om.n_nodes, dtype=torch.float32, device="cuda")
            capi.chns_mg_vcycle(mg, dev(r, torch.float32), z, capi.FP32, op=capi.MG_SHIFTED)
            assert relerr(z.double().cpu().numpy(), ref) < 1e-4
    finally:
        capi.chns_mg_destroy(mg)
        gm.close()

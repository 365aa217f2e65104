"""The FP32 Cahn-Hilliard apply with two leaves per thread (CHNS_APPLY_STREAM): meshes of one leaf, a
lone brick, odd numbers of leaves outside bricks and patches with many hanging slots, FP32 and
bfloat16 coefficients, one CTA for all patches; against the oracle's matrix on the same rounded
inputs and against the CTA-per-patch kernel.

Bounds: as for the other FP32 applies with two leaves per thread, 1e-5 against the oracle (chains
of about 20 roundings of 6e-8, sums of up to about 30 terms). The two kernels differ in the order of
their sums only: 4e-6, twice the bound of the one-component operators for the two terms that add
up in each row."""
import numpy as np
import pytest

from gpu_common import PRM, bf16_round, dev, f32_round, fields, oracle_operator, relerr
from test_gpu_pair_apply import MESHES

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402
from oracle.mesh import Mesh as OMesh  # noqa: E402


def _run(gm, coef, x, prec, kernel):
    capi.chns_mesh_set_apply_config(gm.handle, kernel, 1 if kernel == capi.APPLY_STREAM else 0)
    y = torch.full((x.numel(),), 7.0, dtype=torch.float32, device="cuda")
    capi.chns_apply_ch(gm.handle, capi.make_params(PRM), coef, x, y, prec)
    return y.double().cpu().numpy()


@pytest.mark.parametrize("prec", [capi.FP32, capi.FP32_BF16COEF])
@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("extent", [(1.0, 1.0, 1.0), (1.0, 2.0, 0.5)])
def test_pair_apply_ch(name, extent, prec):
    a, l = MESHES[name]()
    om, gm = OMesh(a, l, extent), Mesh(a, l, extent)
    f = fields(om.n_nodes, 21)
    x = f32_round(f["x"][:2].ravel())
    if prec == capi.FP32:
        phi, u = f32_round(f["phi"]), f32_round(f["u"])
        coef = capi.make_coef(dev(phi, torch.float32), [dev(v, torch.float32) for v in u])
    else:
        phi, u = bf16_round(1.0 + f["phi"]) - 1.0, bf16_round(f["u"])
        coef = capi.make_coef(dev(1.0 + phi, torch.bfloat16), [dev(v, torch.bfloat16) for v in u])
    ref = oracle_operator(om, capi.OP_CH, PRM, phi, u) @ x
    xd = dev(x, torch.float32)
    y = _run(gm, coef, xd, prec, capi.APPLY_STREAM)
    assert relerr(y, ref) < 1e-5
    assert relerr(y, _run(gm, coef, xd, prec, capi.APPLY_PATCH)) < 4e-6
    gm.close()


def test_pair_apply_ch_keeps_nan_where_it_belongs():
    """A NaN of phi, u or x reaches the nodes the CTA-per-patch kernel takes it to and no others."""
    gm = Mesh(*MESHES["random_l2_5"]())
    f = fields(gm.n_nodes, 3)
    for which in ("phi", "u", "x"):
        g = {k: f[k].copy() for k in ("phi", "u", "x")}
        (g["phi"] if which == "phi" else g[which][1])[np.flatnonzero(~gm.boundary)[7]] = np.nan
        coef = capi.make_coef(dev(g["phi"], torch.float32), [dev(v, torch.float32) for v in g["u"]])
        xd = dev(g["x"][:2].ravel(), torch.float32)
        y = _run(gm, coef, xd, capi.FP32, capi.APPLY_STREAM)
        assert np.isnan(y).any()
        assert np.array_equal(np.isnan(y), np.isnan(_run(gm, coef, xd, capi.FP32, capi.APPLY_PATCH)))
    gm.close()

"""FP32 momentum solves after another on the same mesh: the Jacobi preconditioner of each comes from its
own coefficients, whichever kernel the solves before it took (the CTA-per-patch one keeps quadrature
data on the mesh, the persistent one evaluates its coefficients). The iterations are those of the same
solve on a mesh of its own, and the oracle's matrix confirms the residual (5 % for its rounding)."""
import numpy as np
import pytest

from gpu_common import LEAVES, PRM, dev, fields, oracle_operator

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402
from oracle.mesh import Mesh as OMesh  # noqa: E402

# viscosity and time step at which diffusion decides the diagonal
DIFFUSIVE = dict(PRM, Re=0.02, dt=5e-2)


def _solve(gm, prm, f, kernel):
    capi.chns_mesh_set_apply_config(gm.handle, kernel, 0)
    coef = capi.make_coef(dev(f["phi"]), [dev(v) for v in f["u"]], dev(f["mu"]))
    x = torch.zeros(3 * gm.n_nodes, dtype=torch.float64, device="cuda")
    b = f["x"].ravel().copy()
    st = capi.chns_krylov_solve(gm.handle, capi.OP_MOMENTUM, capi.make_params(prm), coef, dev(b), x,
                                capi.make_solver(capi.KSP_GMRES, capi.PC_JACOBI, 1e-10, 4000, 30,
                                                 capi.FP32, 1e-4))
    return st, x.cpu().numpy(), b


@pytest.mark.parametrize("first,second", [(capi.APPLY_PATCH, capi.APPLY_AUTO),
                                          (capi.APPLY_AUTO, capi.APPLY_PATCH),
                                          (capi.APPLY_PATCH, capi.APPLY_PATCH)])
def test_preconditioner_is_of_this_solve(first, second):
    leaves, ext = LEAVES["drop_l3_5"]
    a, l = leaves()
    om, gm, own = OMesh(a, l, ext), Mesh(a, l, ext), Mesh(a, l, ext)
    f1, f2 = fields(om.n_nodes, 43), fields(om.n_nodes, 44)
    _solve(gm, PRM, f1, first)
    st, x, b = _solve(gm, DIFFUSIVE, f2, second)
    ref, _, _ = _solve(own, DIFFUSIVE, f2, second)
    # the order of the atomic sums may move the last iteration
    assert abs(st.iterations - ref.iterations) <= 2, (st.iterations, ref.iterations)
    A = oracle_operator(om, capi.OP_MOMENTUM, DIFFUSIVE, f2["phi"], f2["u"], f2["mu"])
    assert np.linalg.norm(b - A @ x) / np.linalg.norm(b) <= 1.05e-10
    gm.close()
    own.close()

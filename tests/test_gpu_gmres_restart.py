"""GMRES on short vectors (the Gram-Schmidt step in one cooperative launch) over several restart
cycles: restart lengths of either parity, one, and cycles cut short by the iteration limit, with
fewer unknowns than CTAs x 3 and with thousands; the iterate after a fixed number of iterations
against a dense-algebra restarted GMRES on the oracle's matrix.

Bound: both are FP64 and differ by rounding, 1e-16 per operation times the growth of the difference
over at most 9 well-conditioned steps; 1e-9 leaves three digits over what sums of 1e4 terms give."""
import numpy as np
import pytest

from gpu_common import PRM, dev, fields, meshes, oracle_operator, relerr

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402


def _gmres(A, b, restart, its):
    """x after `its` steps of right-preconditioned (Jacobi) GMRES from zero, restarted."""
    dinv, x, done = 1.0 / A.diagonal(), np.zeros_like(b), 0
    while done < its:
        r = b - A @ x
        V, H, k = [r / np.linalg.norm(r)], np.zeros((restart + 1, restart)), 0
        while k < restart and done < its:
            w = A @ (dinv * V[k])
            for i in list(range(k + 1)) * 2:
                d = V[i] @ w
                H[i, k] += d
                w = w - d * V[i]
            H[k + 1, k] = np.linalg.norm(w)
            V.append(w / H[k + 1, k])
            k, done = k + 1, done + 1
        e = np.zeros(k + 1)
        e[0] = np.linalg.norm(r)
        y = np.linalg.lstsq(H[:k + 1, :k], e, rcond=None)[0]
        x = x + dinv * (np.array(V[:k]).T @ y)
    return x


@pytest.mark.parametrize("restart,its", [(1, 4), (2, 6), (3, 9), (4, 7), (5, 9), (30, 9)])
@pytest.mark.parametrize("name", ["uniform2", "drop_l3_5"])
def test_restart_cycles(name, restart, its):
    om, gm = meshes(name)
    f = fields(om.n_nodes, 12)
    # a time step at which advection and diffusion count beside the mass term
    prm = dict(PRM, dt=5e-2)
    A = oracle_operator(om, capi.OP_MOMENTUM, prm, f["phi"], f["u"], f["mu"])
    coef = capi.make_coef(dev(f["phi"]), [dev(f["u"][i]) for i in range(3)], dev(f["mu"]))
    b = f["x"].ravel().copy()
    x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    s = capi.make_solver(capi.KSP_GMRES, capi.PC_JACOBI, 1e-30, its, restart)
    st = capi.chns_krylov_solve(gm.handle, capi.OP_MOMENTUM, capi.make_params(prm), coef, dev(b), x,
                                s, check=False)
    assert st.iterations == its
    ref = _gmres(A, b, restart, its)
    assert np.linalg.norm(b - A @ ref) > 1e-9 * np.linalg.norm(b)  # the cycles have work to do
    assert relerr(x.cpu().numpy(), ref) < 1e-9

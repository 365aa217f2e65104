"""The velocity right-hand sides of a constant state are exact: at constant phi, velocity and pressure
without advection every interpolated value is the constant itself, so that each interior node
receives the cell volume times the constant, with no rounding for numbers that are short sums of
powers of two (density 1 or 1/2, time step 2^-10, Froude number 4, power-of-two cells)."""
import numpy as np
import pytest

from chns_workloads import octree
from gpu_common import PRM, dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402

V = np.array([0.75, -0.5, 1.25])


@pytest.mark.parametrize("phase", [1.0, -1.0])
@pytest.mark.parametrize("extent", [(1.0, 1.0, 1.0), (1.0, 2.0, 0.5)])
@pytest.mark.parametrize("level", [1, 3])
def test_constant_state(level, extent, phase):
    gm = Mesh(*octree.uniform(level), extent)
    n, inner = gm.n_nodes, ~gm.boundary
    prm = capi.make_params(dict(PRM, rho_ratio=2.0, dt=2.0 ** -10, Fr=4.0))
    rho, cell = (1.0 if phase > 0 else 0.5), np.prod(extent) * 8.0 ** -level
    const = lambda a: dev(np.full(n, a))  # noqa: E731
    coef = capi.make_coef(const(phase), [const(0.0)] * 3, const(0.0))
    v, p = [const(a) for a in V], const(0.25)
    out = torch.empty(3 * n, dtype=torch.float64, device="cuda")

    capi.chns_rhs_momentum(gm.handle, prm, coef, v, p, out)
    y = out.cpu().numpy().reshape(3, n)
    for i in range(3):
        expect = cell * rho * (V[i] * 1024.0 - (0.25 if i == 1 else 0.0))
        assert np.array_equal(y[i], np.where(inner, expect, 0.0)), i

    # component 1 has the gravity residual times tau_m, which is no short number
    capi.chns_rhs_velocity_update(gm.handle, prm, coef, v, v, p, p, out)
    y = out.cpu().numpy().reshape(3, n)
    for i in (0, 2):
        assert np.array_equal(y[i], np.where(inner, cell * rho * V[i], 0.0)), i
    gm.close()

"""The Cahn-Hilliard residual of a pure phase at rest (phi = 1 or -1, mu = 0, u = 0) is exactly zero on
every mesh: phi^3 - phi and all differences vanish without rounding, so that a Newton iteration
with any tolerance stops before its first solve."""
import numpy as np
import pytest

from gpu_common import PRM, SMALL, dev, meshes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import capi  # noqa: E402


@pytest.mark.parametrize("phase", [1.0, -1.0])
@pytest.mark.parametrize("name", SMALL)
def test_pure_phase_has_no_residual(name, phase):
    _, gm = meshes(name)
    n = gm.n_nodes
    phi, zero = dev(np.full(n, phase)), dev(np.zeros(n))
    f = torch.full((2 * n,), 7.0, dtype=torch.float64, device="cuda")
    capi.chns_residual_ch(gm.handle, capi.make_params(PRM), phi, zero, phi, zero, [zero] * 3, f)
    assert not f.any()

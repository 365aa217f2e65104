"""GMRES where the one-launch Gram-Schmidt step cannot run: a context that may use less of the device
refuses its cooperative launch (from the first one on, or from a later one, with a column still in
flight), and a grid barrier that timed out. The library is linked with a stand-in for the launch call
that returns the refusal, or sets the mark that a CTA sets whose wait ran out.

The refused solve takes the separate kernels: the iterations and the iterate of the ordinary one,
1e-9 as between GMRES and its restatement on the host (test_gpu_gmres_restart.py)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gpu_common import LEAVES, PRM, dev, fields, relerr

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2107_05123_gb300 import _lib, capi  # noqa: E402
from paper_2107_05123_gb300 import build as b  # noqa: E402
from paper_2107_05123_gb300.session import Mesh  # noqa: E402

FAKE = r"""
#include <cuda_runtime.h>
extern "C" {
int fake_refuse_from = -1, fake_timeout_at = -1, fake_calls = 0;
cudaError_t fake_cooperative_launch(const void* f, dim3 grid, dim3 block, void** args, size_t smem,
                                    cudaStream_t s) {
  const int call = fake_calls++;
  if (fake_refuse_from >= 0 && call >= fake_refuse_from) return cudaErrorCooperativeLaunchTooLarge;
  const cudaError_t e = cudaLaunchCooperativeKernel(f, grid, block, args, smem, s);
  if (e == cudaSuccess && call == fake_timeout_at) {
    double* out = *static_cast<double**>(args[10]);
    return cudaMemsetAsync(out + 63, 1, sizeof(double), s);
  }
  return e;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    """The library with the stand-in, bound like the real one."""
    b.build()
    d = tmp_path_factory.mktemp("fallback")
    (d / "fake.cu").write_text(FAKE)
    nvcc, inc = b._nvcc(), ["-I", b.CSRC]
    subprocess.run([nvcc, *b.ARCH, *b.FLAGS, *inc, "-c", str(d / "fake.cu"), "-o", str(d / "fake.o")],
                   check=True, capture_output=True)
    subprocess.run([nvcc, *b.ARCH, *b.FLAGS, *inc, "-c", os.path.join(b.CSRC, "krylov.cu"), "-o",
                    str(d / "krylov.o"), "-DcudaLaunchCooperativeKernel=fake_cooperative_launch"],
                   check=True, capture_output=True)
    objs = [os.path.join(b.BUILD, os.path.basename(s) + ".o") for s in b.sources()
            if os.path.basename(s) != "krylov.cu"]
    out = str(d / "libchns_fake.so")
    subprocess.run([nvcc, *b.ARCH, "-shared", "-cudart", "static", "-o", out, *objs,
                    str(d / "krylov.o"), str(d / "fake.o"), "-Xcompiler", "-pthread"],
                   check=True, capture_output=True)
    path, _lib.LIB_PATH = _lib.LIB_PATH, out
    try:
        return _lib._load()
    finally:
        _lib.LIB_PATH = path


def _solve(lib, monkeypatch, restart, its, refuse=-1, timeout=-1, check=False):
    monkeypatch.setattr(_lib, "LIB", lib)
    for name, v in (("fake_refuse_from", refuse), ("fake_timeout_at", timeout), ("fake_calls", 0)):
        ctypes.c_int.in_dll(lib, name).value = v
    leaves, ext = LEAVES["drop_l3_5"]
    gm = Mesh(*leaves(), ext)
    f = fields(gm.n_nodes, 12)
    coef = capi.make_coef(dev(f["phi"]), [dev(v) for v in f["u"]], dev(f["mu"]))
    x = torch.zeros(3 * gm.n_nodes, dtype=torch.float64, device="cuda")
    s = capi.make_solver(capi.KSP_GMRES, capi.PC_JACOBI, 1e-30, its, restart)
    try:
        st = capi.chns_krylov_solve(gm.handle, capi.OP_MOMENTUM, capi.make_params(dict(PRM, dt=5e-2)),
                                    coef, dev(f["x"].ravel()), x, s, check=check)
        return st, x.cpu().numpy(), ctypes.c_int.in_dll(lib, "fake_calls").value
    finally:
        gm.close()


@pytest.mark.parametrize("refuse", [0, 1, 4, 6])
@pytest.mark.parametrize("restart,its", [(3, 8), (5, 9), (30, 9)])
def test_refused_launch(lib, monkeypatch, restart, its, refuse):
    st, x, calls = _solve(lib, monkeypatch, restart, its)
    assert st.iterations == its and calls >= its
    st2, x2, calls2 = _solve(lib, monkeypatch, restart, its, refuse=refuse)
    assert calls2 == refuse + 1  # the first refusal is the last launch tried
    assert st2.iterations == its and st2.status == st.status
    assert relerr(x2, x) < 1e-9


@pytest.mark.parametrize("at", [0, 3])
def test_barrier_timeout_is_reported_as_such(lib, monkeypatch, at):
    with pytest.raises(_lib.ChnsError, match="timed out") as e:
        _solve(lib, monkeypatch, 30, 9, timeout=at, check=True)
    assert e.value.status == capi.ECUDA

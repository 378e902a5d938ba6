"""What the library's host code owes its caller on a GPU: how it waits, what a
failed call leaves behind, what it needs of device memory."""
import os
import subprocess
import sys

import pytest

import microstructure as ms

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_BLOCKING = """
import ctypes, time
cu = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(dev, 4) == 0     # blocking synchronisation
import torch
import microstructure as ms
from paper_2003_07720_gb300 import rpm
torch.cuda.init()
with rpm.Context(ms.cell_sphere32(32)) as ctx:
    st, first = ctx.solve(ms.unit_strain(0))
    torch.cuda._sleep(800_000_000)                        # some 0.4 s ahead of the solve
    wall, cpu = time.perf_counter(), time.thread_time()
    st, info = ctx.solve(ms.unit_strain(0))
    wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
assert info["converged"] and info["mean_stress"] == first["mean_stress"]
print(wall, cpu)
"""


def test_solve_sleeps_where_the_device_is_set_to_blocking_synchronisation():
    """The flags are the process's, so the solve runs in a child.  A thread that
    sleeps until its first residual arrives uses next to no processor time."""
    r = subprocess.run([sys.executable, "-c", _BLOCKING], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    wall, cpu = map(float, r.stdout.split())
    assert wall > 0.2 and cpu < 0.25 * wall, (wall, cpu)


def _cu(name, *args):
    import ctypes
    return getattr(ctypes.CDLL("libcuda.so.1"), name)(*args)


@pytest.mark.parametrize("shape", [(16, 16, 16), (48, 48, 48), (4, 8, 12)])
def test_a_refused_launch_leaves_no_error_behind(shape):
    """A map on a stream whose capture was invalidated is refused; the next call,
    on a sound stream, must not find that error."""
    import ctypes

    import numpy as np
    from paper_2003_07720_gb300 import rpm
    cell = ms.cell_sphere32(16)
    cell = ms.Cell(phase=np.zeros(shape, np.uint8), lam=cell.lam, mu=cell.mu, lam0=cell.lam0,
                   mu0=cell.mu0)
    x = torch.zeros((6,) + shape, device="cuda")
    y = torch.empty_like(x)
    E = ms.unit_strain(0)
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert _cu("cuStreamCreate", ctypes.byref(stream), 1) == 0
    with rpm.Context(cell, rpm.rpm_default_options(p_max=0), stream=stream.value) as bad, \
            rpm.Context(cell, rpm.rpm_default_options(p_max=0)) as good:
        torch.cuda.synchronize()
        assert _cu("cuStreamBeginCapture_v2", stream, 2) == 0
        assert _cu("cuStreamSynchronize", stream) != 0        # invalidates the capture
        with pytest.raises(rpm.RpmError):
            bad.apply_gamma(x, E, y)
        assert _cu("cuStreamEndCapture", stream, ctypes.byref(graph)) != 0
        st, info = good.solve(E)
        assert st == rpm.RPM_OK and info["converged"]
    assert _cu("cuStreamDestroy_v2", stream) == 0


@pytest.mark.parametrize("shape,p_max,need", [
    # bytes per context before the reductions took more blocks on small grids
    ((16, 16, 16), 0, 1690016), ((16, 16, 16), 10, 3743136), ((48, 48, 48), 20, 136513296),
    ((24, 96, 48), 40, 242855952), ((64, 64, 64), 20, 322479240), ((1, 64, 64), 250, 53009824)])
def test_a_context_needs_no_more_device_memory_than_it_did(shape, p_max, need):
    """A cap that was enough for a context stays enough."""
    import numpy as np
    from paper_2003_07720_gb300 import rpm
    cell = ms.cell_sphere32(16)
    cell = ms.Cell(phase=np.zeros(shape, np.uint8), lam=cell.lam, mu=cell.mu, lam0=cell.lam0,
                   mu0=cell.mu0)
    with rpm.Context(cell, rpm.rpm_default_options(p_max=p_max, max_device_gb=need / 1e9)) as ctx:
        assert rpm.rpm_device_bytes(ctx.handle) <= need

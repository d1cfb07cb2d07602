"""The units of a mesh do not change how the minimisation is solved: with the
coordinates and the velocities multiplied by a power of two every quantity of a
step scales exactly, so the solver takes the same iterations to the same result.
"""
import numpy as np
import pytest

from paper_1908_05834_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1908_05834_gb300 import build
    build.build()
    from paper_1908_05834_gb300 import bchar
    return bchar


@pytest.mark.parametrize("name,n,log2", [
    ("vortex2d_1024", 48, 8),    # one cluster's system
    ("vortex2d_1024", 48, 10),
    ("vortex2d_1024", 96, 10),   # across the grid
    ("deform3d_128", 12, 8),     # porous, rows of tens of entries
    ("deform3d_128", 12, 12),
])
def test_iterations_do_not_depend_on_the_units(bc, name, n, log2):
    import torch
    wl = inputs.workload(name, n=n)
    dt = (1.0 if len(wl.coords) == 2 else 0.1) / n
    got = []
    for scale in (1.0, 2.0 ** log2):
        coords = [scale * np.asarray(x) for x in wl.coords]
        faces = [scale * u for u in wl.faces(0)]
        mesh = bc.Mesh(coords, wl.phi, bc.default_options())
        mesh.set_velocity(faces)
        c = torch.tensor(wl.c0, dtype=torch.float64, device="cuda")
        out = torch.empty_like(c)
        info = mesh.step(dt, c, out)
        assert info["qp_converged"] == 1
        got.append((info["ip_iters"], info["cg_iters"], info["amg_levels"], out))
        mesh.close()
    assert got[0][:3] == got[1][:3]
    assert torch.equal(got[0][3], got[1][3])

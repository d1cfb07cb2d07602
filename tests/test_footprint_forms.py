"""bchar_device_bytes stays within bchar_estimate_device_bytes for both forms of the
minimisation's linear system, near the limits of the rule that chooses between
them, where a row of A meets the estimate's 3^d entries in the mean.
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


@pytest.mark.parametrize("name,n,dt,pairs,precond", [
    ("vortex2d_1024", 48, 200.0 / 48, (6, 12), 1),  # rows of 7 entries in the mean, 7 pairs each: a long time step
    ("deform3d_128", 24, 0.03, (11, 12), 1),        # near the rule's 12 pairs per entry
    ("deform3d_128", 16, 0.05, (13, 40), 1),        # beyond it: rows and columns
    ("deform3d_128", 16, 0.05, (13, 40), 0),        # the Jacobi solver's own vectors, no hierarchy
])
def test_footprint_of_both_forms(bc, name, n, dt, pairs, precond):
    import torch
    wl = inputs.workload(name, n=n)
    opt = bc.default_options(qp_max_refine=2, qp_precond=precond, qp_max_iter=2000)
    mesh = bc.Mesh(wl.coords, wl.phi, opt)
    c = torch.tensor(wl.c0, dtype=torch.float64, device="cuda")
    out = torch.empty_like(c)
    mesh.set_velocity(wl.faces(0))
    info = mesh.step(dt, c, out)
    rows = np.diff(mesh.export_matrix(0)[0]).astype(np.int64)
    assert pairs[0] <= (rows * (rows - 1)).sum() / rows.sum() <= pairs[1]
    assert info["nnz"] <= 3 ** wl.dim * mesh.nc
    mesh.time_stage(0, 1)  # the product with the matrix brings its vectors along
    now, peak = mesh.device_bytes()
    est = bc.estimate_device_bytes(wl.coords, opt)
    mesh.close()
    assert 0 < now <= peak <= est, (now, peak, est)


def test_without_room_for_the_elimination_rows_and_columns_are_kept(bc):
    """With less device memory left than the row-eliminated system takes, but enough for
    the bipartite one, a step still runs, to the same result."""
    import torch
    wl = inputs.workload("deform3d_128", n=40)
    dt = 0.02
    c = torch.tensor(wl.c0, dtype=torch.float64, device="cuda")
    outs = [torch.empty_like(c) for _ in range(2)]
    faces = wl.faces(0)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def step(out):
        before = free()
        with bc.Mesh(wl.coords, wl.phi, bc.default_options()) as mesh:
            mesh.set_velocity(faces)
            info = mesh.step(dt, c, out)
            assert info["qp_converged"] == 1
            return before - free(), mesh.device_bytes()[1]

    step(outs[0])  # what the library's first launches take is taken
    held, peak = step(outs[0])
    hog = torch.empty(free() - (held - (100 << 20)), dtype=torch.uint8, device="cuda")
    try:
        _, less = step(outs[1])
    finally:
        del hog
        torch.cuda.empty_cache()
    assert less < peak - (100 << 20)
    err = (outs[1] - outs[0]).abs().sum() / outs[0].abs().sum()
    assert float(err) <= 1e-5

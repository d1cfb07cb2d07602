"""Every form of the minimisation's linear solver against the oracle: the
hierarchy of one level, one cluster's systems and those across the grid at
their border, with the rows eliminated and as the bipartite system that rows
too wide for the elimination keep.

The bars are those of the parity tests: c within 1e-5 relative L1 (each side
stops its interior point at a scaled constraint residual of 1e-9 or below, and
the minimiser is unique), mass to 1e-12.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
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


def _mesh(name):
    """coords, phi, faces, dt, balls per axis"""
    if name.startswith("uniform"):
        wl = inputs.workload("vortex2d_32", n=int(name.split()[1]))
        return wl.coords, wl.phi, wl.faces(3), wl.dt, 2
    # one wide layer of cells per axis: their images cover up to 260 others.  An even count
    # of cells, because the field's symmetry puts face ties under an odd one.
    before, after = (int(v) for v in name.split()[1:3])
    x = np.concatenate([[0.0], np.cumsum([1.0] * before + [2.9] + [1.0] * after)])
    coords = [x / x[-1]] * 3
    phi = np.random.Generator(np.random.PCG64(1)).uniform(0.1, 0.3, (before + after + 1) ** 3)
    return coords, phi, inputs.deform3d_faces(coords), 0.1, 1


CASES = [
    # name, rows eliminated, unknowns, entries
    ("uniform 5", True, (25, 32), None),               # one level, solved by its inverse
    ("uniform 6", True, (33, 4096), None),             # two levels
    ("uniform 64", True, (4096, 4096), None),          # the largest of one cluster
    ("uniform 65", True, (4097, 5000), None),          # the smallest across the grid
    ("layers 3 4", False, (2, 4096), (1, 40000)),      # bipartite, one cluster
    ("layers 5 6", False, (2, 4096), (40001, 10**9)),  # bipartite, across the grid
]


@pytest.mark.parametrize("name,schur,unknowns,entries", CASES, ids=[c[0].replace(" ", "-") for c in CASES])
def test_solver_paths_match_oracle(bc, name, schur, unknowns, entries):
    import torch
    coords, phi, faces, dt, nb = _mesh(name)
    om = oracle.Mesh(coords, phi, nb=nb)
    c = np.random.Generator(np.random.PCG64(2)).uniform(size=om.nc)
    mesh = bc.Mesh(coords, phi, bc.default_options(balls_per_axis=nb))
    mesh.set_velocity(faces)
    c_in = torch.tensor(c, device="cuda")
    c_out, again = torch.empty_like(c_in), torch.empty_like(c_in)
    info = mesh.step(dt, c_in, c_out)
    # the case is on the side of the rules that it is here for
    rp, cols, vals = mesh.export_matrix(0)
    B = sp.csr_matrix((np.ones(len(cols)), cols, rp), shape=(mesh.nc, mesh.nc))
    length = np.diff(rp)
    per_column = B.T @ length
    assert (per_column.max() <= 8192 and np.sum(length.astype(np.int64) ** 2) <= 12 * len(cols)) == schur
    if entries:
        assert entries[0] <= 2 * len(cols) <= entries[1]
    assert unknowns[0] <= (mesh.nc if schur else 2 * mesh.nc) <= unknowns[1]

    ref = oracle.step(om, faces, dt, c)
    assert info["qp_converged"] == 1
    assert np.abs(c_out.cpu().numpy() - ref["c"]).sum() / np.abs(ref["c"]).sum() <= 1e-5
    assert abs(info["mass_after"] - info["mass_before"]) <= 1e-12 * info["mass_before"]
    mesh.step(dt, c_in, again)
    assert torch.equal(c_out, again)  # every sum in a fixed order
    mesh.close()


def test_jacobi_solver_matches_multigrid(bc):
    """qp_precond = 0: the passes of the interior point around solves that are
    kernels of their own."""
    import torch
    coords, phi, faces, dt, _ = _mesh("uniform 8")
    c_in = torch.tensor(np.random.Generator(np.random.PCG64(2)).uniform(size=64), device="cuda")
    out = []
    for pre in (0, 1):
        mesh = bc.Mesh(coords, phi, bc.default_options(qp_precond=pre))
        mesh.set_velocity(faces)
        o = torch.empty_like(c_in)
        assert mesh.step(dt, c_in, o)["qp_converged"] == 1
        out.append(o.cpu().numpy())
        mesh.close()
    assert np.abs(out[0] - out[1]).sum() <= 1e-5 * np.abs(out[1]).sum()

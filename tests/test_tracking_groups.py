"""Tracking at the edges of its groups: meshes of fewer cells than a group's 32,
of one more, with cells of unequal ball counts, and with fewer balls than a
warp's lanes, against the oracle.

In FP64 both sides evaluate the same expressions but for the order of roundings:
1e-10 of the smallest width, as in the parity tests, with 0.5 % of the balls
allowed to take the other cell of a face tie.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("varying", [False, True], ids=["constant", "varying"])
@pytest.mark.parametrize("shape,nb", [((2, 2), 1), ((5, 5), 2), ((11, 3), 2), ((6, 6), 5), ((7, 9), 3), ((2, 2, 2), 1),
                                      ((3, 5, 2), 2), ((4, 4, 3), 2)])
def test_tracked_balls_of_ragged_groups(bc, shape, nb, varying):
    import torch
    rng = np.random.Generator(np.random.PCG64(sum(shape) + nb))
    # unequal widths: unequal ball counts per cell, of at most 32
    spread = 1.05 if nb * 1.6 >= 32 ** (1 / len(shape)) else 1.6  # (not uniform: symmetry puts ties there)
    coords = []
    for n in shape:
        x = np.concatenate([[0.0], np.cumsum(rng.uniform(1.0, spread, n))])
        coords.append(x / x[-1])
    nc = int(np.prod(shape))
    phi = rng.uniform(0.1, 0.3, nc) if varying else np.full(nc, 0.7)
    om = oracle.Mesh(coords, phi, nb=nb)
    assert oracle.ball_counts(om).max() <= 32
    faces = inputs.vortex2d_faces(coords) if len(shape) == 2 else inputs.deform3d_faces(coords)
    dt = 0.01
    mesh = bc.Mesh(coords, phi, bc.default_options(balls_per_axis=nb))
    mesh.set_velocity(faces)
    c = torch.tensor(rng.uniform(size=nc), device="cuda")
    info = mesh.step(dt, c, torch.empty_like(c))
    pos, rh, off = mesh.export_tracked()
    s = oracle.substep_count(om, faces, dt)
    assert info["substeps"] == s
    ooff, ocen, orh = oracle.track_balls(om, faces, dt, s, np.arange(nc))
    assert np.array_equal(off, ooff)
    h = min(float(np.min(np.diff(x))) for x in coords)
    err = np.maximum(np.max(np.abs(pos - ocen), axis=1), np.abs(rh - orh))
    assert np.mean(err <= 1e-10 * h) >= 0.995
    mesh.close()

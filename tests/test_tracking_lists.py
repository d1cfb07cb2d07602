"""The two ways in which centres are dealt to lanes with constant porosity: by the lists
of a group of 32 cells (FP32; FP64 where every cell holds the least number of balls), and
in ball order (FP64 otherwise), at the edges of groups, chunks and blocks.

FP64 against the oracle as in the tests of ragged groups: 1e-10 of the smallest width,
0.5 % of the balls may take the other cell of a face tie.  FP32 against FP64: a stage
rounds a local coordinate of at most 1 a dozen times, 12 x 4 stages x 6e-8 per substep,
and an error grows by less than e over the step: 1e-5 of the largest width per substep.
"""
import numpy as np
import pytest

import oracle
from paper_1908_05834_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [((2, 2), 2), ((5, 5), 2), ((11, 11), 2), ((8, 8), 2), ((13, 13), 1), ((3, 3, 3), 2), ((4, 4, 4), 2)]  # cubes: counts from the widths alone


def _problem(shape, spread):
    rng = np.random.Generator(np.random.PCG64(sum(shape)))
    coords = []
    for n in shape:
        x = np.concatenate([[0.0], np.cumsum(rng.uniform(1.0, spread, n))])
        coords.append(x / x[-1])
    faces = inputs.vortex2d_faces(coords) if len(shape) == 2 else inputs.deform3d_faces(coords)
    return coords, np.full(int(np.prod(shape)), 0.7), faces


def _tracked(coords, phi, faces, nb, precision, dt):
    import torch
    from paper_1908_05834_gb300 import build
    build.build()
    from paper_1908_05834_gb300 import bchar
    with bchar.Mesh(coords, phi, bchar.default_options(balls_per_axis=nb, precision=precision, qp_max_refine=0)) as mesh:
        mesh.set_velocity(faces)
        c = torch.zeros(mesh.nc, dtype=torch.float64, device="cuda")
        info = mesh.step(dt, c, torch.empty_like(c))
        return (*mesh.export_tracked(), info["substeps"])


@pytest.mark.parametrize("shape,nb", SHAPES)
def test_equal_counts_by_lists_in_fp64(shape, nb):
    coords, phi, faces = _problem(shape, 1.05)
    om = oracle.Mesh(coords, phi, nb=nb)
    assert np.all(oracle.ball_counts(om) == nb ** len(shape))
    pos, rh, off, s = _tracked(coords, phi, faces, nb, 0, 0.01)
    ooff, ocen, orh = oracle.track_balls(om, faces, 0.01, s, np.arange(om.nc))
    assert np.array_equal(off, ooff)
    h = min(float(np.min(np.diff(x))) for x in coords)
    err = np.maximum(np.max(np.abs(pos - ocen), axis=1), np.abs(rh - orh))
    assert np.mean(err <= 1e-10 * h) >= 0.995


@pytest.mark.parametrize("spread", [1.05, 1.6])
@pytest.mark.parametrize("shape,nb", SHAPES)
def test_fp32_lists_follow_fp64(shape, nb, spread):
    coords, phi, faces = _problem(shape, spread)
    pos, rh, off, s = _tracked(coords, phi, faces, nb, 0, 0.01)
    pos32, rh32, off32, s32 = _tracked(coords, phi, faces, nb, 1, 0.01)
    assert s == s32 and np.array_equal(off, off32)
    h = max(float(np.max(np.diff(x))) for x in coords)
    err = np.maximum(np.max(np.abs(pos - pos32), axis=1), np.abs(rh - rh32))
    assert np.mean(err <= 1e-5 * s * h) >= 0.995

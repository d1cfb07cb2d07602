"""The minimisation's inexact solves leave no more error in c than solves to the
result's accuracy would.  The oracle's minimisation, with exact solves, gets the
step's own scaled matrix, so that only the minimisation differs.

The bar: the last corrector solves go down to a constraint residual of 1e-2 qp_tol
= 1e-11 of each target (the oracle's to 1e-12); and an entry at distance d from its
bounds is held off by the mean complementarity of at most 1e-12 where the iteration
stops, 1e-12 / d of a factor 1 + x.  c is a mean of such factors times c: its relative
L1 error is at most 1e-11 + 1e-12 / d, with the smallest d.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_1908_05834_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cfl", [(24, 1.0), (32, 0.32), (32, 2.0), (64, 2.0)])
def test_minimisation_error_against_exact_solves(n, cfl):
    import torch
    from paper_1908_05834_gb300 import build
    build.build()
    from paper_1908_05834_gb300 import bchar
    wl = inputs.workload("vortex2d_32", n=n)
    volphi = oracle.Mesh(wl.coords, wl.phi).volphi()
    for centre in ((0.4, 0.6), (0.55, 0.35)):
        c0 = inputs.indicator_ball_average(wl.coords, centre, 0.15, 4)
        with bchar.Mesh(wl.coords, wl.phi, bchar.default_options()) as mesh:
            mesh.set_velocity([0.7 * u for u in wl.faces(0)])
            c = torch.tensor(c0, dtype=torch.float64, device="cuda")
            out = torch.empty_like(c)
            assert mesh.step(cfl / n, c, out)["qp_converged"] == 1
            got = out.cpu().numpy()
            A0, AN = (sp.csr_matrix((v, j, p), shape=(mesh.nc, mesh.nc))
                      for p, j, v in (mesh.export_matrix(k) for k in (0, 1)))
        b, _ = oracle.balanced_targets(A0, volphi)
        Aq = AN.copy()
        factor = oracle.minimise(AN, b, volphi)[0]
        Aq.data = AN.data * factor
        distance = max(float(np.minimum(factor, 2.0 - factor).min()), 1e-12)
        ref = oracle.column_fix(Aq, AN, volphi) @ c0 / volphi
        assert np.abs(got - ref).sum() <= (1e-11 + 1e-12 / distance) * np.abs(ref).sum()

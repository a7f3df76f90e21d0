"""Pivots whose squared modulus is beyond 2^1022, where its reciprocal is subnormal: lengths
scaled by 2^-251 scale the operator by 2^502 and its inverse by 2^-502.

Tolerance 1e-12 relative to the field in ordinary units: a subnormal reciprocal near 2^-1024
keeps 50 bits, an error of 2^-51 in each pivot's inverse, over fewer than 200 nodes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402

DEV = "cuda:0"


# one small front; warp and block fronts; pivot blocks of large fronts
@pytest.mark.parametrize("nx,ny", [(4, 4), (9, 11)])
@pytest.mark.parametrize("leaf", [16, 128])
@pytest.mark.parametrize("pivoting", [0, 1])
def test_inverse_scales_with_the_operator(nx, ny, leaf, pivoting):
    import paper_2509_20801_gb300 as g
    eps = torch.ones((nx, ny), dtype=torch.float64, device=DEV)
    v = torch.from_numpy(W.random_vector(nx * ny, seed=nx)[0]).to(DEV)
    z = []
    for scale in (1.0, 2.0 ** -251):
        # sixteen nodes a wavelength: |diagonal| = 984.5 2^502 or 2^511.94; an absorber too weak to raise it
        s = g.Solver(nx, ny, scale / 16, scale / 16, scale, eps, npml=(1,) * 4, pml_R=0.99, nsub=1, overlap=1,
                     interface_pml=1)
        g.stdd_set_option(s.ctx, g.STDD_OPT_PIVOTING, pivoting)
        g.stdd_set_option(s.ctx, g.STDD_OPT_LEAF, leaf)
        s.factor()
        out = torch.empty_like(v)
        g.stdd_apply_preconditioner(s.ctx, v, out)
        z.append(out.cpu().numpy())
        s.close()
    assert np.linalg.norm(z[1] * 2.0 ** 502 - z[0]) <= 1e-12 * np.linalg.norm(z[0])

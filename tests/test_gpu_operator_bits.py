"""The operator and the residual outside the PML, bit for bit, against their sums in the order
documented at the kernel, each product-sum rounded once (exact rationals): k0^2 eps - (-x) -
(+x) - (-y) - (+y) couplings for the diagonal, the diagonal's product, the neighbours -x, +x, -y,
+y, and the right-hand side minus that."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle.fdfd import Problem  # noqa: E402

DEV = "cuda:0"


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


# walks of one column and of several; blocks of 128 rows and a remainder
@pytest.mark.parametrize("nx,ny", [(24, 40), (40, 130), (4000, 260)])
def test_bits_outside_the_pml(nx, ny):
    import paper_2509_20801_gb300 as g
    npml = 4
    w = W.random_medium(nx, ny, ppw=16, seed=7, npml=npml, nsub=1, overlap=1, interface_pml=1)
    P = Problem.from_workload(w)
    k0sq, c = float(P.k0) * float(P.k0), 1.0 / (w.dx * w.dx)
    assert c == 256.0 and w.dx == w.dy
    x, b = (W.random_vector(w.n, seed=k)[0].reshape(nx, ny) for k in (1, 2))
    xd, bd = torch.from_numpy(x).to(DEV), torch.from_numpy(b).to(DEV)
    y, r = torch.empty_like(xd), torch.empty_like(xd)
    s = g.Solver.from_workload(w, eps=torch.from_numpy(w.eps_node).to(DEV))
    g.stdd_apply_operator(s.ctx, xd, y)
    g.stdd_residual(s.ctx, xd, bd, r)
    s.close()
    y, r = y.cpu().numpy(), r.cpu().numpy()
    rng = np.random.default_rng(nx)
    inner_x, inner_y = range(npml + 1, nx - npml - 1), range(npml + 1, ny - npml - 1)
    for _ in range(400):
        i, j = int(rng.choice(inner_x)), int(rng.choice(inner_y))
        d = _fma(k0sq, w.eps_node[i, j], -c) - c - c - c
        parts = []
        for f in (np.real, np.imag):
            v = d * float(f(x[i, j]))
            for a in (x[i - 1, j], x[i + 1, j], x[i, j - 1], x[i, j + 1]):
                v = _fma(c, float(f(a)), v)
            parts.append(v)
        want = complex(*parts)
        assert y[i, j] == want
        assert r[i, j] == complex(b[i, j].real - want.real, b[i, j].imag - want.imag)

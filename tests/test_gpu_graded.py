"""Fields that decay through a box by many orders of magnitude: inside a metal (eps < 0) every
node's value is accurate relative to itself, not only to the largest in the box.

Reference: the band of the stretched operator eliminated without pivoting in numpy's extended
precision.  Tolerance 1e-10, the bar of the local solves, here at every node: sums and factors
err by FP64's unit relative to their own terms, which in a metal have one magnitude at each
depth.  (The update of large fronts runs on the FP64 pipe here; its split products err relative
to their rows' and columns' largest entries.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle.fdfd import Problem  # noqa: E402

DEV = "cuda:0"


def _band_solve(A, b, half):
    n = A.shape[0]
    band = np.zeros((n, 2 * half + 1), np.clongdouble)
    C = A.tocoo()
    band[C.row, C.col - C.row + half] = C.data
    x = b.astype(np.clongdouble)
    for k in range(n):
        m = min(half, n - 1 - k)
        up = band[k, half + 1:half + 1 + m]
        for r in range(k + 1, k + 1 + m):
            f = band[r, k - r + half]
            if f != 0:
                f = f / band[k, half]
                band[r, k - r + half + 1:k - r + half + 1 + m] -= f * up
                x[r] -= f * x[k]
    for k in range(n - 1, -1, -1):
        m = min(half, n - 1 - k)
        x[k] = (x[k] - (band[k, half + 1:half + 1 + m] * x[k + 1:k + 1 + m]).sum()) / band[k, half]
    return x


@pytest.mark.parametrize("nx,ny,eps,along_y", [(24, 24, -40.0, True), (24, 24, -40.0, False), (40, 40, -12.0, True),
                                               (40, 40, -12.0, False), (70, 30, -6.0, False)])
@pytest.mark.parametrize("pivoting", [0, 1])
def test_field_inside_a_metal_is_accurate_at_every_depth(nx, ny, eps, along_y, pivoting):
    import paper_2509_20801_gb300 as g
    w = W.random_medium(nx, ny, ppw=16, seed=3, npml=4, nsub=1, overlap=1, interface_pml=1)
    w.eps_node = np.ones((nx, ny))
    w.eps_node[(slice(None), slice(ny // 3, None)) if along_y else slice(nx // 3, None)] = eps
    b = np.zeros((nx, ny), complex)
    b[(nx // 2, ny // 6) if along_y else (nx // 6, ny // 2)] = 1.0
    ref = _band_solve(Problem.from_workload(w).A, b.ravel(), ny)
    s = g.Solver.from_workload(w, eps=torch.from_numpy(w.eps_node).to(DEV))
    g.stdd_set_option(s.ctx, g.STDD_OPT_PIVOTING, pivoting)
    g.stdd_set_option(s.ctx, g.STDD_OPT_FP64_TC, 0)
    s.factor()
    z = torch.empty(nx * ny, dtype=torch.complex128, device=DEV)
    g.stdd_apply_preconditioner(s.ctx, torch.from_numpy(b.ravel()).to(DEV), z)   # one strip: the whole inverse
    s.close()
    size = np.abs(ref).astype(float)
    assert size.min() < 1e-14 * size.max()
    assert (np.abs(z.cpu().numpy() - ref) / np.abs(ref)).max() <= 1e-10

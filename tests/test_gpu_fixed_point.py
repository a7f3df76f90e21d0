"""complex128 substitutions on fixed-point factors (tensor-core digit products): boxes and
fronts at the edges of the 16- and 32-row tiles and 32-column chains, vectors of widely
different magnitude, exact scaling, and non-finite input.

Tolerance against the oracle: 1e-10, the bar of the local solves (another elimination order
and no pivoting against SuperLU); the products themselves are within 2^-58 of a row's and a
vector chain's largest entries."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle.fdfd import Problem  # noqa: E402
from oracle.stddm import DDM  # noqa: E402

DEV = "cuda:0"


def _problem(nx, ny, nsub, npml, seed=5):
    w = W.random_medium(nx, ny, ppw=16, seed=seed, npml=npml, nsub=nsub, overlap=3, interface_pml=npml)
    return w, DDM.from_workload(w, Problem.from_workload(w))


def _apply(s, v):
    from paper_2509_20801_gb300 import stdd_apply_preconditioner
    z = torch.empty_like(v)
    stdd_apply_preconditioner(s.ctx, v, z)
    return z


def _solver(w, **opts):
    import paper_2509_20801_gb300 as g
    s = g.Solver.from_workload(w, eps=torch.from_numpy(w.eps_node).to(DEV))
    for k, val in opts.items():
        g.stdd_set_option(s.ctx, getattr(g, k), val)
    s.factor()
    return s


# one front; a root of 16 / 17 pivots; chains of 31..33 columns; two strips, odd heights
@pytest.mark.parametrize("nx,ny,nsub,npml", [(5, 5, 1, 1), (9, 11, 1, 2), (16, 40, 1, 3), (33, 17, 1, 4),
                                             (64, 33, 2, 5), (131, 97, 2, 8)])
@pytest.mark.parametrize("pivoting", [0, 1])
def test_boxes_at_tile_edges_match_oracle(nx, ny, nsub, npml, pivoting):
    w, D = _problem(nx, ny, nsub, npml)
    s = _solver(w, STDD_OPT_PIVOTING=pivoting)
    rng = np.random.default_rng(nx)
    for spread in (0, 12):      # entries of one magnitude, entries over twelve decades
        v = W.random_vector(nx * ny, seed=nx + ny)[0] * 10.0 ** (-spread * rng.random(nx * ny))
        z = _apply(s, torch.from_numpy(v).to(DEV)).cpu().numpy()
        ref = D.apply_Minv(v)
        assert np.linalg.norm(z - ref) <= 1e-10 * np.linalg.norm(ref)
    s.close()


def test_powers_of_two_scale_exactly():
    w, _ = _problem(64, 33, 2, 5)
    s = _solver(w)
    v = torch.from_numpy(W.random_vector(w.n, seed=2)[0]).to(DEV)
    z = _apply(s, v)
    for k in (-300, -7, 300):
        assert torch.equal(_apply(s, v * 2.0 ** k), z * 2.0 ** k)
    s.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_vectors_stay_nonfinite_and_leave_nothing_behind(bad):
    w, _ = _problem(64, 33, 2, 5)
    s = _solver(w)
    v = torch.from_numpy(W.random_vector(w.n, seed=2)[0]).to(DEV)
    z = _apply(s, v)
    broken = v.clone()
    broken[w.n // 3] = bad
    assert not torch.isfinite(torch.view_as_real(_apply(s, broken))).all()
    assert torch.equal(_apply(s, v), z)
    s.close()

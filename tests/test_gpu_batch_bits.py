"""A right-hand side's field and residual history do not depend on which others are solved with
it, nor on when those converge: on a grid large enough that the Gram-Schmidt sums of one, eight
or seventeen right-hand sides would be cut into different chunks if the batch set their number
(more than 512 nodes for each of the chunks a single one may have)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("precision,order,count", [(0, 0, 17), (1, 2, 8)])
def test_batch_equals_single_on_a_large_grid(precision, order, count):
    import paper_2509_20801_gb300 as g
    w = W.random_medium(400, 300, ppw=16, seed=31, npml=10, nsub=3, overlap=5, interface_pml=10)
    s = g.Solver.from_workload(w, eps=torch.from_numpy(w.eps_node).to(DEV), precision=precision)
    g.stdd_set_option(s.ctx, g.STDD_OPT_ORDER, order)
    s.factor()
    # dense fields and points: they converge at different steps
    b = torch.zeros((count, w.nx, w.ny), dtype=torch.complex128, device=DEV)
    for k in range(count):
        if k % 2:
            b[k, 30 + 20 * k % 340, 40 + 13 * k % 220] = 1.0 + k
        else:
            b[k] = torch.from_numpy(W.random_vector(w.n, seed=k)[0].reshape(w.nx, w.ny)).to(DEV)
    x, x1 = torch.empty_like(b), torch.empty_like(b[:1])
    opts = dict(restart=12, rtol=1e-7, maxit=400)
    s.set_sources(b)
    s.solve(x, **opts)
    history = [s.history(k) for k in range(count)]
    assert len({len(h) for h in history}) > 1     # some left the batch before others
    for k in sorted({0, 1, count // 2, count - 2, count - 1}):
        s.set_sources(b[k:k + 1].clone())
        s.solve(x1, **opts)
        assert torch.equal(x1[0], x[k])
        assert np.array_equal(s.history(0), history[k])
    s.close()

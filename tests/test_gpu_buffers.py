"""Operator and residual on the caller's own device buffers, and on ones the kernels cannot
use in place (output over the input, shifted over it, off by half an entry): every case gives
the same bits.  Right-hand sides beyond one launch's batch: each as if solved alone."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from oracle.fdfd import Problem  # noqa: E402

DEV = "cuda:0"


def _lib(name, ctx, *ptrs):
    from paper_2509_20801_gb300 import binding
    assert getattr(binding.lib, name)(ctx, *ptrs, 1) == 0


# odd sizes: one block of rows, remainders of 128-row blocks, walks of several columns
@pytest.mark.parametrize("nx,ny", [(5, 5), (64, 127), (41, 129), (1600, 1030)])
def test_operator_and_residual_same_bits_in_every_buffer(nx, ny):
    import paper_2509_20801_gb300 as g
    w = W.random_medium(nx, ny, ppw=16, seed=3, npml=1 if nx == 5 else 10, nsub=1, overlap=1, interface_pml=1)
    A = Problem.from_workload(w).A
    s = g.Solver.from_workload(w, eps=torch.from_numpy(w.eps_node).to(DEV))
    n = w.n
    xh, bh = (W.random_vector(n, seed=k)[0] for k in (1, 2))
    x, b = torch.from_numpy(xh).to(DEV), torch.from_numpy(bh).to(DEV)
    y, r = torch.empty_like(x), torch.empty_like(x)
    g.stdd_apply_operator(s.ctx, x, y)
    rel = g.stdd_residual(s.ctx, x, b, r)
    ref = A @ xh    # 1e-13 of the largest entry: five products and a sum per entry, two orders of adding
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
    assert np.abs(r.cpu().numpy() - (bh - ref)).max() <= 1e-13 * np.abs(bh - ref).max()

    both = torch.zeros(3 * n + 8, dtype=torch.complex128, device=DEV)
    def at(offset_bytes, v=None):
        raw = both.view(torch.float64).view(torch.uint8)[offset_bytes:offset_bytes + 16 * n]
        if v is not None:
            raw.copy_(v.view(torch.float64).view(torch.uint8))
        return raw, ctypes.c_void_p(raw.data_ptr())
    def value(raw):
        return raw.clone().view(torch.float64).view(torch.complex128)
    for xo, yo in ((0, 0), (0, 16 * (n // 2)), (16 * (n // 2), 0), (8, 16 * (n + 1)), (0, 16 * n + 8)):
        _, px = at(xo, x)
        out, py = at(yo)
        _lib("stdd_apply_operator", s.ctx, px, py)
        assert torch.equal(value(out), y)
    for xo, bo, ro in ((0, 16 * n, 16 * n), (0, 16 * n, 0), (0, 16 * n, 16 * (n // 2)), (8, 16 * n + 32, 16 * n + 32),
                       (0, 16 * n, 32 * n + 8), (0, 0, 16 * n)):
        _, pb = at(bo, b)
        _, px = at(xo, x)
        out, pr = at(ro)
        got = ctypes.c_double()
        _lib("stdd_residual", s.ctx, px, pb, pr, ctypes.byref(got))
        if xo == bo:
            assert np.abs(value(out).cpu().numpy() - (xh - ref)).max() <= 1e-13 * np.abs(xh - ref).max()
        else:
            assert torch.equal(value(out), r) and got.value == rel
    s.close()


@pytest.mark.parametrize("order", [0, 1, 2])
def test_seventeen_right_hand_sides_equal_singles(order):
    import paper_2509_20801_gb300 as g
    w = W.random_medium(90, 41, ppw=16, seed=9, npml=8, nsub=3, overlap=4, interface_pml=6)
    s = g.Solver.from_workload(w, eps=torch.from_numpy(w.eps_node).to(DEV))
    g.stdd_set_option(s.ctx, g.STDD_OPT_ORDER, order)
    s.factor()
    b = torch.from_numpy(np.stack([W.random_vector(w.n, seed=k)[0].reshape(w.nx, w.ny) for k in range(17)])).to(DEV)
    x, x1 = torch.empty_like(b), torch.empty_like(b[:1])
    s.set_sources(b)
    s.solve(x, restart=8, rtol=1e-9, maxit=400)
    for k in (0, 15, 16):
        s.set_sources(b[k:k + 1].clone())
        s.solve(x1, restart=8, rtol=1e-9, maxit=400)
        assert torch.equal(x1[0], x[k])
    s.close()

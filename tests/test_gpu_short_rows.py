"""Readouts of boxes with short rows: the same values, and no more time than rows that fill a block."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from oracle import grad_ref  # noqa: E402
from paper_1909_13412_gb300 import lbp  # noqa: E402
from paper_1909_13412_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def device(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("nx,ny,nz", [(1, 9, 17), (2, 11, 7), (31, 3, 5), (127, 2, 3), (128, 3, 2), (129, 3, 4), (260, 1, 3)])
def test_f0_gradient_of_any_row_length(nx, ny, nz):
    """Against the FP64 reference, within the bound of the adjoint's other tests."""
    n, steps = 2, 5
    ps = wl.uniform_particles(n, (nz, ny, nx), 10.0, 0.5, 0.26, 1e-4, 5, 6)
    f0 = wl.perturbed_populations(oracle.d3q15()[1], (nz, ny, nx), 0.02, 4)
    g = np.random.default_rng(3).standard_normal((steps, n, 3))
    t = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), requires_grad=True)
    x = t(f0)
    V, _, _ = grad_ref.run(x, t(ps.r), t(ps.V), t(ps.M), t(ps.gamma), t(ps.R), t(0.8), steps)
    (torch.tensor(g) * V).sum().backward()
    want = x.grad.numpy().reshape(15, -1)
    h = lbp.lbp_create(nx, ny, nz, 0.8)
    lbp.lbp_set_populations(h, np.ascontiguousarray(f0))
    lbp.lbp_particles_add(h, ps.r, ps.V, ps.M, ps.gamma, ps.R)
    lbp.lbp_adjoint_record(h, steps, 2)
    got = np.empty((15, h.N))
    lbp.lbp_adjoint_backward(h, steps, g, None, {"f0": got})
    lbp.lbp_destroy(h)
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()


def seconds(f):
    best = np.inf
    for _ in range(6):  # the first is a warm-up
        torch.cuda.synchronize()
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


def test_short_rows_cost_no_more():
    """The same bytes, as contiguous: within a factor of three (with a block per
    row segment, rows of one node took thirty times as long)."""
    fields, f0 = [], []
    for nx, m in ((1, 2000), (128, 177)):
        h = lbp.lbp_create(nx, m, m, 0.8)
        rho, u = device(h.N), device(3, h.N)
        fields.append(seconds(lambda: [lbp.lbp_read_fields(h, rho, u) for _ in range(10)]) / 10)
        ps = wl.uniform_particles(1, (m, m, nx), 10.0, 0.5, 0.26, 1e-4, 5, 6)
        lbp.lbp_particles_add(h, ps.r, ps.V, ps.M, ps.gamma, ps.R)
        lbp.lbp_adjoint_record(h, 1, 1)
        g = torch.ones((1, 1, 3), dtype=torch.float64, device="cuda")
        grads = {"v0": device(1, 3)}
        without = seconds(lambda: lbp.lbp_adjoint_backward(h, 1, g, None, grads))
        grads["f0"] = device(15, h.N)
        f0.append(seconds(lambda: lbp.lbp_adjoint_backward(h, 1, g, None, grads)) - without)
        lbp.lbp_destroy(h)
    assert fields[0] <= 3 * fields[1]
    assert f0[0] <= 3 * max(f0[1], 1e-4)

"""What calls other than steps leave of a handle's state."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1909_13412_gb300 import lbp  # noqa: E402
from paper_1909_13412_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def handle(shape, n, precision=lbp.LBP_F32, stream=None, kT=1e-4):
    nx, ny, nz = shape
    h = lbp.lbp_create(nx, ny, nz, 0.8, precision=precision, stream=stream)
    if n:
        ps = wl.uniform_particles(n, (nz, ny, nx), 10.0, 0.5, 0.26, 1e-3, 5, 6)
        lbp.lbp_particles_add(h, ps.r, ps.V * 30, ps.M, ps.gamma, ps.R)
        lbp.lbp_particles_set_params(h, kT=kT, seed=3)
    return h


def state(h):
    n = h.np
    out = [np.empty((15, h.N))] + [np.empty((n, 3)) for _ in range(4)]
    lbp.lbp_read_populations(h, out[0])
    if n:
        lbp.lbp_particles_read(h, *out[1:])
    return out


def same(a, b):
    return len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("chain", [True, False])
def test_backward_leaves_the_conservation_budget(chain):
    """The reverse sweep replays the recorded steps: what F_R and F_ext put in was
    counted when they were recorded."""
    h = handle((20, 18, 16), 30)
    lbp.lbp_set_use_graphs(h, chain)
    lbp.lbp_particles_set_external_force(h, np.full((30, 3), 1e-5))
    lbp.lbp_budget_track(h)
    lbp.lbp_adjoint_record(h, 12, 5)
    before = lbp.lbp_budget(h)
    lbp.lbp_adjoint_backward(h, 12, np.ones((12, 30, 3)), None, {"v0": np.empty((30, 3))})
    assert np.array_equal(lbp.lbp_budget(h), before) and before[7:].any()
    lbp.lbp_destroy(h)


@pytest.mark.parametrize("warm", [0, 3])
@pytest.mark.parametrize("n", [0, 5])
def test_steps_refuse_to_be_captured(n, warm):
    """A replay would not advance the host's buffer parity and step index.  The
    capture itself stays valid, and the handle goes on as if not called."""
    st = torch.cuda.Stream()
    h, twin = (handle((24, 16, 12), n, stream=s) for s in (st, None))
    for k in (h, twin):
        if warm:
            lbp.lbp_step(k, warm)
    x = torch.zeros(4, device="cuda")
    v = torch.empty((3, n, 3), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    calls = [lambda: lbp.lbp_step(h, 1), lambda: lbp.lbp_step(h, 2), lambda: lbp.lbp_step_exchange(h),
             lambda: lbp.lbp_autotune(h, 1)]
    if n:
        calls += [lambda: lbp.lbp_adjoint_record(h, 3, 1, v), lambda: lbp.lbp_step_exchange(h, v[0], v[1], v[2])]
    with torch.cuda.graph(g, stream=st):
        x.add_(1)
        for call in calls:
            with pytest.raises(lbp.LbpError) as ei:
                call()
            assert ei.value.status == lbp.LBP_ESTATE
        lbp.lbp_step(h, 0)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [3.0] * 4
    for k in (h, twin):
        lbp.lbp_step(k, 4)
    assert lbp.lbp_get_step_index(h) == warm + 4
    assert same(state(h), state(twin))
    lbp.lbp_destroy(h)
    lbp.lbp_destroy(twin)


def step_seconds(h, steps=60):
    lbp.lbp_step(h, steps)
    took = []
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        lbp.lbp_step(h, steps)
        torch.cuda.synchronize()
        took.append(time.perf_counter() - t)
    return float(np.median(took)) / steps


@pytest.mark.parametrize("shape,n", [((66, 64, 64), 0), ((34, 32, 32), 1), ((62, 66, 60), 0), ((126, 128, 128), 500)])
@pytest.mark.parametrize("precision", [lbp.LBP_BF16, lbp.LBP_F16])
def test_autotune_picks_the_fastest_step(shape, n, precision):
    """Boxes where the two-node kernel, whose steps are not chained, is as fast as
    the others alone: every pick's step within 15 % of the best one's (the steps
    differ by 20 to 50 % there)."""
    h = handle(shape, n, precision)
    lbp.lbp_step(h, 3)
    picks = {lbp.lbp_autotune(h, 5)[:2] for _ in range(12)}
    took = {}
    for rows, variant in [(1, 0), (2, 0), (4, 0), (1, 1), (2, 1)]:
        lbp.lbp_set_block_shape(h, rows, variant)
        took[rows, variant] = step_seconds(h)
    for pick in picks:
        assert took.get(pick, np.inf) <= 1.15 * min(took.values()), (pick, took)
    lbp.lbp_destroy(h)


@pytest.mark.parametrize("shape,n,precision", [((66, 24, 20), 0, lbp.LBP_F16), ((34, 32, 32), 40, lbp.LBP_BF16), ((62, 20, 24), 2, lbp.LBP_F16),
                                               ((3, 5, 130), 60, lbp.LBP_F32), ((32, 24, 16), 9, lbp.LBP_F32)])
def test_autotune_leaves_the_handle(shape, n, precision):
    """Also where whole steps are timed: a tuned handle goes on as its twin, with the
    correlator, the conservation budget and the error flag as they were."""
    out = []
    for tune in (True, False):
        h = handle(shape, n, precision)
        lbp.lbp_budget_track(h)
        if n:
            lbp.lbp_vacf_configure(h, 20)
        lbp.lbp_step(h, 7)
        before = lbp.lbp_budget(h), lbp.lbp_diagnostics(h)["overflow_shares"], lbp.lbp_get_step_index(h)
        if tune:
            for _ in range(8):
                lbp.lbp_autotune(h, 3)
                after = lbp.lbp_budget(h), lbp.lbp_diagnostics(h)["overflow_shares"], lbp.lbp_get_step_index(h)
                assert np.array_equal(before[0], after[0]) and before[1:] == after[1:]
        lbp.lbp_check(h)
        lbp.lbp_step(h, 80)
        res = state(h)
        if n:
            res += [np.empty(21), np.empty(21, np.int64)]
            lbp.lbp_vacf_read(h, *res[-2:])
        lbp.lbp_check(h)
        lbp.lbp_destroy(h)
        out.append(res)
    assert same(*out)


def gradient(h, steps, every, precision=lbp.LBP_F32):
    n = h.np
    lbp.lbp_adjoint_record(h, steps, every)
    g = np.random.default_rng(1).standard_normal((steps, n, 3))
    out = {"tau": np.empty(1), "v0": np.empty((n, 3)), "gamma": np.empty(n)}
    lbp.lbp_adjoint_backward(h, steps, g, None, out)
    return list(out.values())


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


MB = 1 << 20


def test_gradient_memory_is_reused_and_released():
    """A second gradient takes no more memory and a much smaller one gives the large
    blocks back; lbp_adjoint_release gives back what is kept, with the recording."""
    h = handle((64, 64, 64), 6)
    copy = 64 ** 3 * 60  # bytes of the populations
    lbp.lbp_step(h, 2)
    start = free_bytes()
    gradient(h, 30, 30)
    one = free_bytes()
    assert start - one >= 30 * copy  # a checkpoint and 29 states, at least
    gradient(h, 30, 30)
    assert free_bytes() == one
    gradient(h, 4, 4)
    assert free_bytes() >= one + 20 * copy
    lbp.lbp_adjoint_release(h)
    assert free_bytes() >= start - 2 * MB
    with pytest.raises(lbp.LbpError) as ei:
        lbp.lbp_adjoint_backward(h, 4, np.ones((4, 6, 3)), None, {"v0": np.empty((6, 3))})
    assert ei.value.status == lbp.LBP_ESTATE
    twin = handle((64, 64, 64), 6)  # the same state reached without the gradients in between
    lbp.lbp_step(twin, 2 + 30 + 30 + 4)
    assert same(state(h), state(twin))
    assert same(gradient(h, 8, 3), gradient(twin, 8, 3))
    lbp.lbp_destroy(h)
    lbp.lbp_destroy(twin)


def test_gradient_memory_does_not_starve_other_handles():
    """With the device nearly full, a new handle gets the idle block of another's
    reverse sweep, whose next gradient is the same."""
    h, twin = handle((128, 128, 128), 4), handle((128, 128, 128), 4)
    gradient(h, 21, 21)  # keeps about 2.8 GB
    want = gradient(twin, 21, 21), gradient(twin, 21, 21)
    lbp.lbp_destroy(twin)
    torch.cuda.empty_cache()
    filler = torch.empty(free_bytes() - 1536 * MB, dtype=torch.uint8, device="cuda")
    assert free_bytes() < 2000 * MB
    other = lbp.lbp_create(256, 256, 256, 0.8)  # 2 GB
    lbp.lbp_step(other, 1)
    lbp.lbp_check(other)
    lbp.lbp_destroy(other)
    del filler
    torch.cuda.empty_cache()
    assert same(gradient(h, 21, 21), want[1])
    lbp.lbp_destroy(h)

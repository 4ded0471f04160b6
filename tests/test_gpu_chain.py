"""The steps of one call, launched as a chain, against the same steps one call each: bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1909_13412_gb300 import lbp  # noqa: E402
from paper_1909_13412_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


def run(boxes, counts, precision, mode, calls, shape, chain=True, lag=-1):
    h = lbp.lbp_create_batch([(*b, 0.8) for b in boxes], precision=precision)
    if shape is not None:
        lbp.lbp_set_block_shape(h, *shape)
    lbp.lbp_set_use_graphs(h, chain)
    for k, ((nx, ny, nz), n) in enumerate(zip(boxes, counts)):
        if n:
            ps = wl.uniform_particles(n, (nz, ny, nx), 10.0, 0.5, 0.26, 1e-3, 5 + k, 6 + k)
            lbp.lbp_particles_add_to(h, k, ps.r, ps.V * 30, ps.M, ps.gamma, ps.R)
    lbp.lbp_particles_set_params(h, kT=1e-3, seed=3, mode=mode)
    if lag >= 0:
        lbp.lbp_vacf_configure(h, lag)
    for n in calls:
        lbp.lbp_step(h, n)
    n = sum(counts)
    out = [np.empty(15 * h.N)] + [np.empty((n, 3)) for _ in range(4)]
    lbp.lbp_read_populations(h, out[0])
    lbp.lbp_particles_read(h, *out[1:])
    if lag >= 0:
        out += [np.empty(lag + 1), np.empty(lag + 1, np.int64)]
        lbp.lbp_vacf_read(h, *out[-2:])
    lbp.lbp_check(h)
    lbp.lbp_destroy(h)
    return out


@pytest.mark.parametrize("boxes,counts", [
    ([(32, 32, 32)], [1]),              # a few marked rows
    ([(3, 5, 131)], [40]),              # corners that wrap in every direction, records that overflow
    ([(260, 9, 8)], [300]),             # three segments a row, most rows marked
    ([(128, 80, 72)], [500]),           # more row segments than resident warps of the four-node kernel
    ([(33, 21, 19), (32, 7, 9), (5, 4, 3)], [9, 3, 1]),  # short rows
    ([(96, 64, 64)], [9000]),           # enough particles for the other order of preparation
    ([(64, 64, 64)], [20000]),          # more particle blocks than are resident at a time
    ([(64, 20, 20), (17, 9, 30), (130, 8, 8)], [2, 0, 30])])
@pytest.mark.parametrize("precision,shape", [
    (lbp.LBP_F32, None), (lbp.LBP_F32, (1, 0)), (lbp.LBP_F32, (4, 0)), (lbp.LBP_BF16, (2, 0)), (lbp.LBP_F16, None), (lbp.LBP_F16, (2, 1)),
    (lbp.LBP_BF16, None)])
def test_steps_of_one_call_equal_single_calls(boxes, counts, precision, shape):
    if shape == (2, 1) and any(b[0] % 2 for b in boxes):
        pytest.skip("two nodes per thread need even rows")
    want = run(boxes, counts, precision, lbp.LBP_STOKESLET, [1] * 40, shape, chain=False)
    for calls in ([40], [7, 33]):
        got = run(boxes, counts, precision, lbp.LBP_STOKESLET, calls, shape)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("mode", [lbp.LBP_POINTWISE, lbp.LBP_BROWNIAN])
def test_chained_modes_and_correlator_blocks(mode):
    args = ([(40, 36, 34)], [50], lbp.LBP_F32, mode)
    want = run(*args, [1] * 150, None, chain=False, lag=30)
    got = run(*args, [150], None, lag=30)
    assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("boxes,counts", [
    ([(100, 60, 36)], [200]),           # more row segments than resident blocks: marks
    ([(32, 16, 16)], [17]),             # a partial second block of particles, no marks
    ([(64, 63, 61)], [40]),             # an odd number of rows
    ([(64, 40, 40), (130, 9, 8)], [30, 0])])
@pytest.mark.parametrize("precision", [lbp.LBP_F32, lbp.LBP_F16])
def test_chained_adjoint_equals_plain_launches(boxes, counts, precision):
    """Replay and reverse sweep as a chain against ordinary launches, bit for bit (no record overflows)."""
    out = []
    for chain in (True, False):
        h = lbp.lbp_create_batch([(*b, 0.8) for b in boxes], precision=precision)
        lbp.lbp_set_use_graphs(h, chain)
        n, steps = sum(counts), 23
        for k, ((nx, ny, nz), m) in enumerate(zip(boxes, counts)):
            if m:
                ps = wl.uniform_particles(m, (nz, ny, nx), 10.0, 0.5, 0.26, 1e-3, 5 + k, 6 + k)
                lbp.lbp_particles_add_to(h, k, ps.r, ps.V * 30, ps.M, ps.gamma, ps.R)
        lbp.lbp_particles_set_params(h, kT=1e-3, seed=3)
        v, r = np.empty((steps, n, 3)), np.empty((steps, n, 3))
        lbp.lbp_adjoint_record(h, steps, 9, v, r)
        g = np.random.default_rng(1)
        grads = {"tau": np.empty(len(boxes)), "kT": np.empty(1), "gamma": np.empty(n), "radius": np.empty(n),
                 "mass": np.empty(n), "v0": np.empty((n, 3)), "r0": np.empty((n, 3)), "f0": np.empty((15, h.N))}
        lbp.lbp_adjoint_backward(h, steps, g.standard_normal((steps, n, 3)), None, grads)
        lbp.lbp_check(h)
        lbp.lbp_destroy(h)
        out.append([v, r, *grads.values()])
    assert all(np.array_equal(a, b) for a, b in zip(*out))
    assert np.abs(out[0][-1]).max() > 0

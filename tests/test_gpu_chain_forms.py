"""Chained steps without particles, and with the couplings that mark differently, against single calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
from paper_1909_13412_gb300 import lbp  # noqa: E402
from paper_1909_13412_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu
W = oracle.d3q15()[1]


def run(boxes, n, precision, calls, shape=None, chain=True, mode=lbp.LBP_STOKESLET, lag=-1, body=None):
    h = lbp.lbp_create_batch([(*b, 0.7) for b in boxes], precision=precision)
    if shape is not None:
        lbp.lbp_set_block_shape(h, *shape)
    lbp.lbp_set_use_graphs(h, chain)
    f = [wl.perturbed_populations(W, b[::-1], 0.02, 3 + k).reshape(15, -1) for k, b in enumerate(boxes)]
    lbp.lbp_set_populations(h, np.concatenate(f, 1))
    if n:
        ps = wl.uniform_particles(n, boxes[0][::-1], 10.0, 0.5, 0.26, 1e-3, 5, 6)
        lbp.lbp_particles_add(h, ps.r, ps.V, ps.M, ps.gamma, ps.R)
        lbp.lbp_particles_set_params(h, kT=1e-3, seed=3, mode=mode)
        if lag >= 0:
            lbp.lbp_vacf_configure(h, lag)
    if body is not None:
        lbp.lbp_set_body_force(h, body)
    for k in calls:
        lbp.lbp_step(h, k)
    out = [np.empty((15, h.N)), np.empty((3, h.N))]
    lbp.lbp_read_populations(h, out[0])
    lbp.lbp_read_fields(h, None, out[1])
    if n:
        out += [np.empty((n, 3)) for _ in range(4)]
        lbp.lbp_particles_read(h, *out[-4:])
    if lag >= 0:
        out += [np.empty(lag + 1), np.empty(lag + 1, np.int64)]
        lbp.lbp_vacf_read(h, *out[-2:])
    lbp.lbp_check(h)
    lbp.lbp_destroy(h)
    return out


@pytest.mark.parametrize("boxes", [
    [(1, 1, 1)], [(3, 5, 131)], [(32, 32, 32)], [(260, 9, 8)],
    [(66, 63, 61)],                 # more blocks than are resident at a time
    [(33, 21, 19), (32, 7, 9), (5, 4, 3)]])
@pytest.mark.parametrize("precision,shape", [
    (lbp.LBP_F32, None), (lbp.LBP_F32, (1, 0)), (lbp.LBP_F32, (4, 0)), (lbp.LBP_BF16, None), (lbp.LBP_BF16, (1, 0)),
    (lbp.LBP_BF16, (2, 0)), (lbp.LBP_BF16, (4, 0)), (lbp.LBP_F16, None), (lbp.LBP_F16, (1, 0)), (lbp.LBP_F16, (2, 0))])
def test_chained_steps_without_particles(boxes, precision, shape):
    args = (boxes, 0, precision)
    kw = {"shape": shape, "body": (1e-6, -2e-6, 3e-6)}
    want = run(*args, [1] * 31, chain=False, **kw)
    for calls in ([31], [8, 23]):
        assert all(np.array_equal(a, b) for a, b in zip(run(*args, calls, **kw), want))


@pytest.mark.parametrize("boxes,precision,shape", [
    ([(64, 64, 64)], lbp.LBP_F32, None), ([(64, 64, 64)], lbp.LBP_F32, (1, 0)), ([(100, 96, 60)], lbp.LBP_F32, (4, 0)),
    ([(128, 80, 72)], lbp.LBP_F16, None), ([(63, 64, 64)], lbp.LBP_BF16, None), ([(128, 160, 72)], lbp.LBP_BF16, (2, 3)),
    ([(128, 160, 120)], lbp.LBP_F16, (4, 3)), ([(128, 130, 120)], lbp.LBP_F32, (1, 0)), ([(150, 130, 120)], lbp.LBP_F32, (1, 0))])
@pytest.mark.parametrize("mode", [lbp.LBP_STOKESLET, lbp.LBP_POINTWISE, lbp.LBP_BROWNIAN])
@pytest.mark.parametrize("n", [1, 60, 1500])
def test_chained_couplings_on_marked_boxes(boxes, precision, shape, mode, n):
    """Boxes beyond the marks' thresholds and, with four rows, on both sides of the
    particle count above which there are none; a correlator block ends inside."""
    args = (boxes, n, precision)
    want = run(*args, [1] * 70, shape=shape, chain=False, mode=mode, lag=20)
    got = run(*args, [70], shape=shape, mode=mode, lag=20)
    assert all(np.array_equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("boxes", [[(16, 10, 8), (24, 6, 10)], [(24, 3, 5)], [(136, 6, 6)]])
@pytest.mark.parametrize("precision", [lbp.LBP_BF16, lbp.LBP_F16])
def test_dense_forces_on_every_shape(boxes, precision):
    """Several times more force shares than the records hold: every kernel takes its
    segments' overflow (the two- and four-node ones pairs of it at a time)."""
    n = 20 * boxes[0][1] * boxes[0][2] // 8
    want = run(boxes, n, precision, [12], (1, 0), chain=False)
    shapes = [(2, 0), (1, 1), (2, 1), (4, 1), (1, 2), (1, 3), (2, 3), (4, 3)]
    for shape in shapes:
        got = run(boxes, n, precision, [12], shape)
        assert all(np.array_equal(a, b) for a, b in zip(got, want)), shape

"""The FP64 readouts (populations, moments) against the plain FP64 evaluation, bit for bit.

The kernels form the moments in integers and widen FP32 values on their bits;
values that do not fit those forms take FP64 instructions.  Stored bit patterns
of every kind go in through a checkpoint: ordinary deviations, ranges too wide
for the integer split, zeros, denormals, infinities and NaNs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_1909_13412_gb300 import lbp  # noqa: E402

pytestmark = pytest.mark.gpu

E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 1),
              (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)])
W = np.array([2.0 / 9.0] + [1.0 / 9.0] * 6 + [1.0 / 72.0] * 8)
HEADER = 128  # bytes before the stored planes of a checkpoint


def stored_values(kind, precision, count, rng):
    """(raw stored words, their FP32 values before any scale) of `count` populations."""
    v = rng.standard_normal(count) * 1e-3
    if kind == "wide":
        v *= np.exp2(rng.integers(-30, 4, count).astype(float))
    elif kind == "special":
        v *= np.exp2(rng.integers(-130, 120, count).astype(float))
        v[rng.random(count) < 0.3] = 0.0
        v[rng.random(count) < 0.1] = -0.0
        for x in (np.inf, -np.inf, np.nan, 3.4e38, 1e-45):
            v[rng.random(count) < 0.002] = x
    with np.errstate(over="ignore"):
        f = v.astype(np.float32)
        if precision == lbp.LBP_F16:
            raw = (f * np.float32(1024 * 9)).astype(np.float16)
            return raw.view(np.uint16), raw.astype(np.float32)
    bits = f.view(np.uint32)
    if precision == lbp.LBP_BF16:
        return (bits >> 16).astype(np.uint16), (bits & 0xFFFF0000).astype(np.uint32).view(np.float32)
    return bits, f


@pytest.mark.parametrize("kind", ["ordinary", "wide", "special"])
@pytest.mark.parametrize("precision", [lbp.LBP_F32, lbp.LBP_BF16, lbp.LBP_F16])
@pytest.mark.parametrize("boxes", [[(131, 5, 3)], [(1, 2, 9), (128, 3, 2), (260, 1, 3)]])
def test_readouts_equal_the_fp64_evaluation(boxes, precision, kind):
    rng = np.random.default_rng([len(boxes), precision, len(kind)])
    h = lbp.lbp_create_batch([(*b, 0.8) for b in boxes], precision=precision)
    raw, g = stored_values(kind, precision, 15 * h.N, rng)
    buf = lbp.lbp_checkpoint_save(h)
    buf[HEADER:] = raw.view(np.uint8)
    lbp.lbp_checkpoint_load(h, buf)
    g = g.reshape(15, h.N)
    with np.errstate(all="ignore"):
        if precision == lbp.LBP_F16:
            g = g * (W.astype(np.float32) * np.float32(1.0 / 1024.0))[:, None]
        g = g.astype(np.float64)
        f = torch.empty(15 * h.N, dtype=torch.float64, device="cuda")
        lbp.lbp_read_populations(h, f)
        assert np.array_equal(f.cpu().numpy().reshape(15, -1), W[:, None] + g, equal_nan=True)
        rho, u, p = np.empty(h.N), np.empty((3, h.N)), np.empty(h.N)
        lbp.lbp_read_fields(h, rho, u, p)
        drho, want = np.zeros(h.N), np.zeros((3, h.N))
        at = 0
        for nx, ny, nz in boxes:
            n = nx * ny * nz
            for a in range(15):
                v = np.roll(g[a, at:at + n].reshape(nz, ny, nx), E[a][::-1], (0, 1, 2)).reshape(-1)
                drho[at:at + n] += v
                for k in range(3):
                    want[k, at:at + n] += E[a][k] * v
            at += n
        assert np.array_equal(rho, 1.0 + drho, equal_nan=True)
        assert np.array_equal(u, want, equal_nan=True)
        assert np.array_equal(p, (1.0 + drho) / 3.0, equal_nan=True)
    lbp.lbp_destroy(h)

"""Errors of the double-float quotient, root, reciprocal and half-slope on the
device, against exact arithmetic.

Bounds, set before the first run: the errors of the same operations built on IEEE
binary32 reciprocals and roots with double-float remainders, emulated with binary32
on the host over 16 million operands of 1 to 2 and e^-3 to e^3 (root mean square,
and the largest with a tenth added, as the largest of two samples differ)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N = 1 << 21
BOUNDS = {"df64_quotient": (3.17e-15, 3.5e-14), "df64_sqrt": (1.50e-15, 1.45e-14), "df64_rcp": (2.37e-15, 1.7e-14),
          "df64_half_slope": (3.64e-15, 3.5e-14)}


def operands(seed):
    rng = np.random.default_rng(seed)
    x = np.where(rng.random(N) < 0.5, rng.uniform(1, 2, N), np.exp(rng.uniform(-3, 3, N)))
    hi = x.astype(np.float32)
    return hi.astype(np.float64) + (x - hi).astype(np.float32)       # exact as a pair


@pytest.mark.parametrize("op", sorted(BOUNDS))
def test_error(op):
    from paper_2012_02925_gb300._binding import check_face_op
    a, b = operands(1), operands(2)
    out = check_face_op(op, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    # the residual of the result in a wide type: h = hi + lo, h b - a and so on
    A, B, h = (x.astype(np.longdouble) for x in (a, b, out[:, 0]))
    h = h + out[:, 1]
    if op == "df64_quotient":
        err = (h * B - A) / A
    elif op == "df64_rcp":
        err = h * A - 1
    elif op == "df64_sqrt":
        err = (h * h - A) / (2 * A)
    else:
        err = (h * (A + B) - A * B) / (A * B)
    err = np.abs(err).astype(np.float64)
    rms, worst = np.sqrt((err ** 2).mean()), err.max()
    assert rms <= BOUNDS[op][0] and worst <= BOUNDS[op][1], (rms, worst)

"""The fixed-point Roe flux, integer slope and integer quotient as the device
evaluates them (its own approximate reciprocals, roots and inline instructions):
the flux's error against 113-bit arithmetic, component by component, within the
bound of the host build's (tests/test_fixed_roe_accuracy.py); the same faces taken;
slope and quotient within one unit in the last place of the exact value."""
import math
from fractions import Fraction

import numpy as np
import pytest

from test_fixed_roe_accuracy import compile_fluxes, faces, no_worse

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N = 4000


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return compile_fluxes(tmp_path_factory.mktemp("device_accuracy"))


def device(x, **kw):
    from paper_2012_02925_gb300._binding import check_roe64
    out = check_roe64(torch.from_numpy(np.ascontiguousarray(x)).cuda(), **kw).cpu().numpy()
    return np.where(out[:, :1] == 1.0, out[:, 1:], np.nan)


@pytest.mark.parametrize("fix_all", [0, 1])
@pytest.mark.parametrize("jump", [0.0, 1e-3, 0.1])
@pytest.mark.parametrize("mach", [1e-6, 1e-3, 0.05, 0.5, 1.0, 2.0, 4.0, 7.9])
def test_flux_no_less_accurate_than_binary64(host, mach, jump, fix_all):
    rng = np.random.default_rng(21)
    for axis in (False, True):
        x = faces(rng, N, mach, jump, axis=axis)
        got = device(x, fix_all=fix_all)
        no_worse(host(x, fix_all=fix_all, given=got), N, 0.9)
        # the scales come from approximations: a face at the very edge may differ
        assert (np.isnan(got[:, 0]) != np.isnan(host(x, fix_all=fix_all)[1][:, 0])).mean() < 1e-3


def test_flux_refuses_what_does_not_fit(host):
    base = np.array([1.0, 0.3, 0.2, 0.1, 0.7, 1.0, 0.3, 0.2, 0.1, 0.7, 1.0, 0.0, 0.0, 1.0])
    rows = []
    for at, bad in [(0, np.nan), (0, np.inf), (0, 0.0), (0, -1.0), (5, 8.0), (4, np.nan), (9, -1.0), (4, 1e300),
                    (1, np.inf), (7, np.nan), (2, 200.0), (10, np.nan), (10, 2.5), (13, 0.0), (13, np.nan)]:
        rows.append(base.copy())
        rows[-1][at] = bad
    assert np.isnan(device(np.array(rows))).all()
    assert np.isfinite(device(base[None])).all()


def pairs():
    rng = np.random.default_rng(22)
    edge = [1.0, 2.0, 1.0 - 2.0 ** -53, 2.0 - 2.0 ** -52, 1.5, 1.0 + 2.0 ** -52]
    p = [(a * 2.0 ** i, b) for a in edge for b in edge for i in (0, 1, 10, 53, 62, 63, 64, 70)]
    p += list(zip(rng.uniform(0.5, 2, 4000) * 2.0 ** rng.integers(-40, 40, 4000), rng.uniform(0.5, 2, 4000)))
    return np.array(p + [(-a, -b) for a, b in p])


@pytest.mark.parametrize("op", ["quotient", "half_slope"])
def test_integer_quotients(op):
    from paper_2012_02925_gb300._binding import check_face_op
    p = pairs()
    a, b = (torch.from_numpy(np.ascontiguousarray(np.abs(p[:, i]) if op == "quotient" and i else p[:, i])).cuda() for i in (0, 1))
    got = check_face_op(op, a, b).cpu().numpy()[:, 0]
    for x, y, g in zip(a.cpu().tolist(), b.cpu().tolist(), got.tolist()):
        X, Y = Fraction(x), Fraction(y)
        want = X / Y if op == "quotient" else X * Y / (X + Y)
        assert abs(Fraction(g) - want) <= Fraction(float(np.spacing(abs(float(want))))), (x, y, g)


def test_integer_quotients_of_special_values():
    from paper_2012_02925_gb300._binding import check_face_op
    inf, nan = math.inf, math.nan

    def run(op, table):
        t = torch.tensor([r[:2] for r in table], dtype=torch.float64, device="cuda")
        return check_face_op(op, t[:, 0].contiguous(), t[:, 1].contiguous()).cpu().numpy()[:, 0], [r[2] for r in table]

    for op, table in (("half_slope", [(nan, -1.0, nan), (-1.0, nan, nan), (nan, 1.0, nan), (inf, -1.0, 0.0),
                                      (inf, 1.0, nan), (1.0, -1.0, 0.0), (0.0, 1.0, 0.0), (4e-31, 4e-31, 0.0)]),
                      ("quotient", [(0.0, 3.0, 0.0), (1e300, 1e-300, inf), (-1e300, 1e-300, -inf), (1e-300, 1e300, 0.0),
                                    (nan, 1.0, nan), (1.0, nan, nan), (1.0, 0.0, nan), (1.0, 1e-310, nan), (1.0, -1.0, nan)])):
        got, want = run(op, table)
        assert np.array_equal(got, np.array(want), equal_nan=True), (op, got)

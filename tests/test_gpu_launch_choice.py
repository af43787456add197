"""What an automatic launch picks, and what a face does that leaves the
fixed-point ranges: the rule gives different shapes and k-chunks for problems of
different extents; blocks in which some, most or all faces take the binary64 flux
(density ratios of up to 36, Mach numbers above 15) agree with the oracle and
bit for bit between tile shapes."""
import numpy as np
import pytest

import cases
import oracle
from test_gpu_parity import TOL_RES, rel_err_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = {
    "plane": lambda: cases.vortex_2d(37),
    "wide_plane": lambda: cases.vortex_2d(700),
    "small": lambda: cases.mms_3d((9, 21, 14)),
    "thin": lambda: cases.mms_3d((70, 33, 2)),
    "ordinary": lambda: cases.mms_3d((96, 64, 80)),
}


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32flux"])
def test_the_rule_tells_problems_apart(prec):
    import paper_2012_02925_gb300 as fv
    picks = {}
    for name, problem in SIZES.items():
        s = fv.Solver.from_problem(problem(), precision=prec)
        assert s.launch()["tile"] == 0 and s.launch()["kchunk"] == 0
        picks[name] = s.launch_choice()
        s.close()
    assert len({p[0] for p in picks.values()}) >= 2, picks
    assert len({p[1] for p in picks.values()}) >= 2, picks
    s = fv.Solver.from_problem(SIZES["small"](), precision=prec, tile=3, kchunk=5)
    assert s.launch_choice() == (3, 5)
    s.close()


def block(kind):
    pb = cases.mms_3d((33, 18, 13), curvilinear=True, with_source=False)
    b = pb.blocks[0]
    q = pb.q.reshape(5, b.nk + 4, b.nj + 4, b.ni + 4)
    rng = np.random.default_rng(9)
    if kind != "fast":       # the same velocity and temperature at another density
        f = 6.0 ** rng.uniform(-1, 1, q.shape[1:])
        if kind == "some":
            f = np.where(rng.random(f.shape) < 0.02, f, 1.0)
        q *= f
    else:
        k = 0.5 * (q[1:4] ** 2).sum(axis=0) / q[0]
        q[1:4] *= 30.0
        q[4] += 899.0 * k
    return pb


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("kind", ["some", "dense", "fast"])
def test_faces_outside_the_fixed_point_ranges(kind, prec):
    import paper_2012_02925_gb300 as fv
    pb = block(kind)
    o = oracle.Oracle(pb)
    ref = o.residual(pb.q.copy())
    out = []
    for tile, kchunk in ((0, 0), (3, 4), (8, 2), (11, 5)) + (((12, 3),) if prec == "fp64" else ()):
        s = fv.Solver.from_problem(pb, precision=prec, tile=tile, kchunk=kchunk)
        s.set_state(torch.from_numpy(pb.q).cuda())
        out.append(s.residual(0).cpu().numpy())
        s.close()
    assert rel_err_fields(out[0], ref, o, pb.q) <= TOL_RES[prec]
    assert all(np.array_equal(out[0], x) for x in out[1:])

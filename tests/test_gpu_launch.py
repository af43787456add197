"""The automatic launch (tile 0, kchunk 0) over problems whose shape or k-chunk
it picks differently: bit-equal to a given tile shape (a face and a cell are
evaluated alike in every tile), with and without physical boundaries."""
import numpy as np
import pytest

import cases

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBLEMS = {
    "vortex": lambda: cases.vortex_2d(37),
    "narrow": lambda: cases.mms_3d((9, 21, 14)),
    "thin": lambda: cases.mms_3d((70, 33, 2)),
    "chunks": lambda: cases.mms_3d((33, 18, 61)),
    "uneven": lambda: cases.multiblock_batched(nblocks=5, lo=5, hi=31, seed=3),
    "inlet": lambda: cases.inlet_2d(104, 32, perturb=0.02, seed=1),
    "ogrid": lambda: cases.ellipse_ogrid(40, 14, 9, perturb=0.02, seed=2),
}


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32flux"])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_bit_equal_to_a_given_tile(name, prec):
    import paper_2012_02925_gb300 as fv
    pb = PROBLEMS[name]()
    out = []
    for tile, kchunk in ((0, 0), (3, 2), (11, 5)) + (((12, 3),) if prec == "fp64" else ()):
        s = fv.Solver.from_problem(pb, precision=prec, tile=tile, kchunk=kchunk)
        s.set_state(torch.from_numpy(pb.q).cuda())
        if pb.source is not None:
            s.set_source(torch.from_numpy(np.concatenate([x.ravel() for x in pb.source])).cuda())
        for _ in range(2):
            s.rk_step(pb.dt)
        out.append(s.get_state(0).cpu().numpy())
        s.close()
    assert np.isfinite(out[0]).all()
    assert all(np.array_equal(out[0], x) for x in out[1:])

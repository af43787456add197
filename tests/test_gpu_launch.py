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


ROW_PROBLEMS = {
    "below": lambda: cases.mms_3d((31, 7, 3)),
    "exact": lambda: cases.mms_3d((32, 8, 2), curvilinear=True),
    "above": lambda: cases.mms_3d((33, 9, 5), curvilinear=True),
    "two": lambda: cases.mms_3d((64, 14, 4)),
    "plane": lambda: cases.inlet_2d(104, 33, perturb=0.02, seed=1),
    "walls": lambda: cases.ellipse_ogrid(64, 16, 7, perturb=0.02, seed=2),
    "laminar": lambda: cases.mms_periodic_3d((33, 15, 5), curvilinear=True, visc=1, mu=0.05),
}


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32flux"])
@pytest.mark.parametrize("name", sorted(ROW_PROBLEMS))
def test_row_shapes_bit_equal_to_a_listed_one(name, prec):
    """Tiles 5 and 8 take their faces by rows of 32 cells, tile 3 from a list:
    the same faces at the edges of tiles and blocks, bit for bit."""
    import paper_2012_02925_gb300 as fv
    if name == "laminar" and prec == "fp32flux":
        pytest.skip("its temperatures are relative to each tile's first cell")
    pb = ROW_PROBLEMS[name]()
    out = []
    for tile, kchunk in ((3, 2), (5, 3), (8, 2)):
        s = fv.Solver.from_problem(pb, precision=prec, tile=tile, kchunk=kchunk)
        s.set_state(torch.from_numpy(pb.q).cuda())
        out.append(s.residual(0).cpu().numpy())
        s.close()
    assert np.isfinite(out[0]).all()
    assert all(np.array_equal(out[0], x) for x in out[1:])


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32flux"])
@pytest.mark.parametrize("name", ["vortex", "inlet", "narrow"])
def test_tile_numbers_without_a_shape(name, prec):
    """12 exists in binary64 only, 13 in 2-D only; these and larger numbers
    run everywhere, bit-equal to 11."""
    import paper_2012_02925_gb300 as fv
    pb = PROBLEMS[name]()
    out = []
    for tile in (11, 12, 13, 99):
        s = fv.Solver.from_problem(pb, precision=prec, tile=tile)
        s.set_state(torch.from_numpy(pb.q).cuda())
        out.append(s.residual(0).cpu().numpy())
        s.close()
    assert np.isfinite(out[0]).all()
    assert all(np.array_equal(out[0], x) for x in out[1:])

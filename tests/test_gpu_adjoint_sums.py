"""The adjoint's sums in binary64 with double-float face sweeps: the cotangents
of the stage input fill binary64's significand.  A sum or a recovery in pairs of
binary32 ends some 48 bits down, and its last bit as a binary64 number is zero
but for a few percent of the values; binary64's is as often one as zero."""
import numpy as np
import pytest

import cases

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBLEMS = {
    "one_block": lambda: cases.mms_3d((14, 11, 9), curvilinear=True, limiter=2, fix_all=1),
    "connected": lambda: cases.multiblock_batched(nblocks=6, lo=5, hi=12, seed=8, limiter=2, fix_all=1),
    "plane": lambda: cases.vortex_2d(24),
}


@pytest.mark.parametrize("arith", ["fp64", "df64"])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_cotangents_fill_the_significand(name, arith):
    import paper_2012_02925_gb300 as fv
    pb = PROBLEMS[name]()
    s = fv.Solver.from_problem(pb, precision="fp64")
    s.set_adjoint_arith(arith)
    lam = torch.from_numpy(np.random.default_rng(3).normal(size=s.field_size)).cuda()
    lam_in, lam_q0 = torch.empty_like(lam), torch.zeros_like(lam)
    s.adjoint_vjp(2, pb.dt, torch.from_numpy(pb.q).cuda(), lam, lam_in, lam_q0)
    x = lam_in.cpu().numpy()
    s.close()
    odd = (x[x != 0].view(np.int64) & 1).mean()
    assert 0.4 < odd < 0.6, odd

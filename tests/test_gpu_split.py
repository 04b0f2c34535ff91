"""One summation order of the hops at every size: the applies to one right-hand side of a small
lattice (the directions of a site on four warps) and to many at once (one warp) give the same
bits."""
import pytest
import torch

from synthetic import gaussian_half5d

from gpu_common import make_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,L,Ls,nrhs", [
    (1, (8, 8, 8, 8), 16, 2), (1, (8, 8, 4, 4), 6, 12), (1, (4, 4, 4, 8), 12, 12), (1, (4, 4, 4, 4), 20, 16),
    (1, (4, 4, 4, 4), 32, 12), (0, (4, 4, 4, 4), 16, 24), (0, (4, 4, 4, 6), 4, 40), (0, (8, 4, 4, 4), 8, 16),
    (0, (4, 4, 4, 8), 10, 12), (0, (4, 4, 4, 4), 24, 12)])
def test_many_right_hand_sides_give_the_bits_of_one(prec, L, Ls, nrhs):
    """The groups of 32 / (Ls / 2) sites of one right-hand side are below the rule's 608 (FP32) or
    456 (FP64), those of all of them above it."""
    from paper_1501_04950_gb300 import dwf
    sysm = make_case(L, Ls, "varying", alpha=1.3, bc_t=-1, black=1)
    op = dwf.DWF(L, Ls, sysm.M5, sysm.m, sysm.alpha, sysm.b, sysm.c, bc_t=-1, rb_parity=1)
    op.load_gauge(torch.from_numpy(sysm.U).cuda())
    groups = -(-(L[0] * L[1] * L[2] * L[3] // 2) // (32 // (Ls // 2)))
    limit = 608 if prec == 1 else 456
    assert groups <= limit < groups * nrhs
    psi = torch.stack([torch.from_numpy(gaussian_half5d(L, Ls, seed=k)) for k in range(2)]).cuda()
    many = psi.repeat(nrhs // 2, 1, 1, 1, 1).contiguous()
    x, y = op.new_field(prec, nrhs), op.new_field(prec, nrhs)
    op.pack_half(x, many, prec, nrhs)
    x1, y1 = op.new_field(prec), op.new_field(prec)
    for fn in (op.apply_Dbb, op.apply_Dbb_dag):
        fn(y, x, prec, nrhs)
        got = y.view(nrhs, -1)
        for k in range(2):
            op.pack_half(x1, psi[k], prec)
            fn(y1, x1, prec)
            for r in range(k, nrhs, 2):
                assert torch.equal(got[r], y1)

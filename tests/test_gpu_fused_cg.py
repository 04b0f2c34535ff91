"""The fused CG steps: their sums, launch order and bits, against the same solve with
other launches (all comparisons bitwise unless a tolerance is stated)."""
import pytest
import torch

from synthetic import gaussian_source4d

from gpu_common import make_case

pytestmark = pytest.mark.gpu


def _op(sysm, **kw):
    from paper_1501_04950_gb300 import dwf
    op = dwf.DWF(sysm.lattice, sysm.Ls, sysm.M5, sysm.m, sysm.alpha, sysm.b, sysm.c,
                 bc_t=int(sysm.bc_t), rb_parity=sysm.black_parity, **kw)
    op.load_gauge(torch.from_numpy(sysm.U).cuda())
    return op


def _solve(sysm, src, nrhs=1, **kw):
    """Propagators and (iterations, FP64 residual) of every source, from a handle of its own."""
    op = _op(sysm, **kw)
    prop = torch.empty_like(src)
    st = op.cgne_solve(src, prop, nrhs=nrhs)
    torch.cuda.synchronize()
    op.close()
    return prop, [(s["iterations"], s["true_resid"]) for s in st]


@pytest.mark.parametrize("prec", [1, 2, 3])
def test_staged_solve_matches_direct_loads(prec, monkeypatch):
    """The norms of the staged kernel, whose CTAs have a fifth warp (the producer), against
    those of the direct-load kernel with CTAs of the same sites (128 threads): exact sums
    (FP32, FP16) and the sum tree (BF16)."""
    sysm = make_case((8, 8, 8, 10), 16, "mobius", alpha=1.2, m=0.1)
    src = torch.from_numpy(gaussian_source4d(sysm.lattice, seed=1)).cuda()
    monkeypatch.setenv("DWF_HOP_TILE", "default")
    direct = _solve(sysm, src, precision_inner=prec)
    monkeypatch.delenv("DWF_HOP_TILE")
    monkeypatch.setenv("DWF_TMA", "1")
    staged = _solve(sysm, src, precision_inner=prec)
    assert staged[1] == direct[1]
    assert torch.equal(torch.view_as_real(staged[0]), torch.view_as_real(direct[0]))

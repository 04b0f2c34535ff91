"""The tuned kernels' dispatch by Ls, size and layout, against the generic kernels, the
oracle or plain torch, at the edges of their tiles.

Tolerances (2-norm of the difference over 2-norm of the reference unless stated): FP64
results 1e-13 (~1e3 roundings of 1.1e-16 a site, which add up like a random walk), FP32
2e-6, FP32 and FP64 sums of ~1e6 terms 1e-13; conversions are exact.
"""
import numpy as np
import pytest
import torch

import oracle as O
from synthetic import gaussian_half5d

from gpu_common import make_case

pytestmark = pytest.mark.gpu


def _op(sysm, **kw):
    from paper_1501_04950_gb300 import dwf
    op = dwf.DWF(sysm.lattice, sysm.Ls, sysm.M5, sysm.m, sysm.alpha, sysm.b, sysm.c,
                 bc_t=int(sysm.bc_t), rb_parity=sysm.black_parity, **kw)
    op.load_gauge(torch.from_numpy(sysm.U).cuda())
    return op


def _rel(a, b):
    return float(torch.linalg.norm(torch.view_as_real(a - b)) / torch.linalg.norm(torch.view_as_real(b)))


def _applies(op, psi, prec, nrhs):
    out = []
    for fn in (op.apply_Dbb, op.apply_Dbb_dag):
        x, y, back = op.new_field(prec, nrhs), op.new_field(prec, nrhs), torch.empty_like(psi)
        op.pack_half(x, psi, prec, nrhs)
        fn(y, x, prec, nrhs)
        op.unpack_half(back, y, prec, nrhs)
        out.append(back)
    return out


@pytest.mark.parametrize("Ls", [4, 6, 10, 12, 20, 24, 32])
@pytest.mark.parametrize("L,nrhs", [((2, 2, 2, 2), 1), ((2, 6, 2, 4), 3), ((8, 8, 8, 8), 1)])
def test_every_compiled_ls_matches_generic(Ls, L, nrhs, monkeypatch):
    """D_bb, D_bb^+ and D_alpha: ragged last CTAs, sites that straddle warps (Ls / 2 not a
    power of two), and both kernels of the choice by size (directions on one warp / four)."""
    sysm = make_case(L, Ls, "varying", alpha=1.4, bc_t=-1, black=1)
    g = torch.Generator(device="cuda").manual_seed(1)
    Vh = int(np.prod(L)) // 2
    psi = torch.view_as_complex(torch.randn(nrhs, Ls, Vh, 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))
    full = torch.view_as_complex(torch.randn(Ls, *L[::-1], 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))
    res = []
    for generic in (True, False):
        if generic:
            monkeypatch.setenv("DWF_GENERIC_KERNELS", "1")
        else:
            monkeypatch.delenv("DWF_GENERIC_KERNELS")
        op = _op(sysm)
        out = torch.empty_like(full)
        op.apply_dalpha(out, full, 0.7, 0.3)
        res.append([_applies(op, psi, prec, nrhs) for prec in (0, 1)] + [[out]])
        op.close()
    for tol, ref, got in zip((1e-13, 2e-6, 1e-13), *res):
        for a, b in zip(got, ref):
            assert _rel(a, b) <= tol


def test_unstable_recurrence_takes_the_dense_inverse():
    """|O_k / D_k| > 1: the cyclic recurrence would amplify rounding by orders of magnitude,
    so such coefficients keep the dense inverse (the oracle's D_bb to 1e-11: the operator
    itself is ill-conditioned there)."""
    L, Ls = (4, 2, 2, 4), 16
    sysm = O.DWFSystem(L, Ls, -1.8, 0.3, 1.3, np.full(Ls, 0.1), np.full(Ls, 3.0), make_case(L, Ls).U)
    op = _op(sysm)
    psi = gaussian_half5d(L, Ls, seed=4)
    got = _applies(op, torch.from_numpy(psi).cuda()[None], 0, 1)[0][0]
    assert _rel(got, torch.from_numpy(sysm.dbb(psi)).cuda()) <= 1e-11


@pytest.mark.parametrize("Ls", [2, 3, 8, 10, 31, 32])
@pytest.mark.parametrize("L", [(2, 2, 2, 2), (6, 2, 4, 2), (4, 10, 2, 6)])
def test_layout_conversions(Ls, L):
    """pack and unpack (exact in FP64) and the full-field split and merge (through D_alpha
    with B = 0 and C = -1 blocks: b = c = 0 leaves no hopping term), odd and even Ls."""
    from paper_1501_04950_gb300 import dwf
    V = int(np.prod(L))
    op = dwf.DWF(L, Ls, -1.8, 0.25, 1.0, np.zeros(Ls), np.zeros(Ls))
    g = torch.Generator(device="cuda").manual_seed(Ls)
    psi = torch.view_as_complex(torch.randn(2, Ls, V // 2, 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))
    x, back = op.new_field(0, 2), torch.zeros_like(psi)
    op.pack_half(x, psi, 0, 2)
    op.unpack_half(back, x, 0, 2)
    assert torch.equal(torch.view_as_real(back), torch.view_as_real(psi))
    # internal layout: [component][pair][re, im][lane]
    n5 = Ls * V // 2
    ref = torch.view_as_real(psi.permute(0, 2, 1, 3, 4).reshape(2, n5 // 2, 2, 12)).permute(0, 3, 1, 4, 2)
    assert torch.equal(x.view(torch.float64).view(2, -1)[:, :24 * n5], ref.reshape(2, -1))
    eye = torch.eye(3, dtype=torch.complex128, device="cuda").expand(*L[::-1], 4, 3, 3).contiguous()
    op.load_gauge(eye)
    full = torch.view_as_complex(torch.randn(Ls, *L[::-1], 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))
    out = torch.empty_like(full)
    op.apply_dalpha(out, full, 1.0, 0.25)
    up, dn = full.roll(-1, 0), full.roll(1, 0)   # psi_{s+1}, psi_{s-1}
    up[-1] *= -0.25
    dn[0] *= -0.25
    ref = full.clone()
    ref[..., 2:, :] -= up[..., 2:, :]
    ref[..., :2, :] -= dn[..., :2, :]
    assert _rel(out, ref) <= 1e-15


@pytest.mark.parametrize("L", [(4, 4, 4, 2), (8, 8, 16, 16), (8, 8, 16, 18), (24, 24, 24, 24)])
def test_reduction_tree(L):
    """S = Re phi^+ X over 4 blocks (one group), 512 (whole groups), 576 (a ragged last group)
    and 2432 (the cap): against a torch dot product of the same fields."""
    from paper_1501_04950_gb300 import dwf
    Ls = 8
    op = dwf.DWF(L, Ls, -1.8, 1.0, 1.0, np.ones(Ls), np.zeros(Ls), rel_tol=1e-3)
    V = int(np.prod(L))
    eye = torch.eye(3, dtype=torch.complex128, device="cuda").expand(*L[::-1], 4, 3, 3).contiguous()
    op.load_gauge(eye)
    g = torch.Generator(device="cuda").manual_seed(7)
    phi = torch.view_as_complex(torch.randn(Ls, V // 2, 4, 3, 2, dtype=torch.float64, device="cuda", generator=g))
    X = torch.empty_like(phi)
    S, _ = op.action(phi, X)
    ref = torch.vdot(phi.reshape(-1), X.reshape(-1)).real.item()
    assert abs(S - ref) <= 1e-13 * abs(ref)


@pytest.mark.parametrize("L,Ls,black,bc_t", [((2, 2, 2, 4), 3, 0, -1), ((4, 2, 2, 2), 5, 1, 1),
                                             ((2, 4, 4, 2), 6, 1, -1), ((4, 4, 2, 2), 16, 0, -1)])
def test_force_matches_oracle(L, Ls, black, bc_t):
    """dS/dU for odd and even Ls, both parities, against the oracle's gradient (1e-12)."""
    sysm = make_case(L, Ls, "varying", alpha=1.2, bc_t=bc_t, black=black)
    op = _op(sysm)
    X = gaussian_half5d(L, Ls, seed=5)
    G = torch.empty(*L[::-1], 4, 3, 3, dtype=torch.complex128, device="cuda")
    Xd = torch.from_numpy(X).cuda()
    op.force(G, Xd, Xd, projected=False)
    ref = torch.from_numpy(O.force_gradient(sysm, X, X)).cuda()
    assert _rel(G, ref) <= 1e-12


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("L,Ls,scale", [((4, 4, 4, 4), 8, 1e-8), ((2, 6, 2, 4), 8, 1e14), ((4, 2, 6, 2), 12, 1.0),
                                        ((8, 8, 8, 8), 16, 1.0)])
def test_cg_sums_match_unfused(L, Ls, scale, prec, monkeypatch):
    """The exact sums of the fused CG (norms of 1e-16 .. 1e28 times the field's, down to 1e-36
    at convergence, near the end of FP32's range, in which the squares of a slice are formed;
    a point source, whose slices differ by many orders of magnitude; ragged CTAs; one and four
    warps a site) against the unfused CG with its tree sums: the same iteration count to one poll
    (the recurrences differ by FP32 rounding only) and the same propagator to 1e-7."""
    from synthetic import point_source4d
    sysm = make_case(L, Ls, "mobius", alpha=1.2, m=0.1)
    src = torch.from_numpy(scale * point_source4d(L, 1, 2)).cuda()
    res = []
    for unfused in (True, False):
        if unfused:
            monkeypatch.setenv("DWF_UNFUSED_CG", "1")
        else:
            monkeypatch.delenv("DWF_UNFUSED_CG")
        op = _op(sysm, precision_inner=prec, check_every=2)
        prop = torch.empty_like(src)
        st = op.cgne_solve(src, prop)[0]
        assert st["true_resid"] <= 1e-10
        res.append((st["iterations"], prop))
        op.close()
    slack = 4 if prec == 1 else 40   # 16-bit recurrences part ways at their replacements
    assert abs(res[0][0] - res[1][0]) <= slack
    assert _rel(res[1][1], res[0][1]) <= 1e-7

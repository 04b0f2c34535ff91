"""Internal half-fields that do not start on a 16-byte boundary (a caller's own buffer with an
offset of one element): the conversions and applies give what they give on aligned fields."""
import pytest
import torch

from synthetic import gaussian_half5d

from gpu_common import make_case

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(torch.linalg.norm(torch.view_as_real(a - b)) / torch.linalg.norm(torch.view_as_real(b)))


@pytest.mark.parametrize("Ls", [7, 8, 10])
@pytest.mark.parametrize("prec,offset,tol", [(0, 8, 1e-13), (1, 4, 2e-6), (1, 8, 2e-6), (2, 4, 1e-2), (3, 4, 5e-2)])
def test_fields_off_the_16_byte_boundary(Ls, prec, offset, tol):
    """pack and unpack move the same bytes; D_bb, its allocation-free form and D_bb^+ agree to the
    roundings by which the generic kernels, which take such fields, differ from the tuned ones."""
    from paper_1501_04950_gb300 import dwf
    sysm = make_case((4, 2, 6, 4), Ls, "varying", alpha=1.3, bc_t=-1, black=1)
    op = dwf.DWF(sysm.lattice, Ls, sysm.M5, sysm.m, sysm.alpha, sysm.b, sysm.c, bc_t=-1, rb_parity=1)
    op.load_gauge(torch.from_numpy(sysm.U).cuda())
    nrhs = 2
    psi = torch.stack([torch.from_numpy(gaussian_half5d(sysm.lattice, Ls, seed=k)) for k in range(nrhs)]).cuda()
    size = op.new_field(prec, nrhs).numel()
    res = []
    for off in (0, offset):
        x, y = [torch.zeros(size + 16, dtype=torch.uint8, device="cuda")[off:off + size] for _ in range(2)]
        assert x.data_ptr() % 16 == off
        op.pack_half(x, psi, prec, nrhs)
        out = [torch.empty_like(psi)]
        op.unpack_half(out[0], x, prec, nrhs)
        for fn in (op.apply_Dbb, op.apply_Dbb_noalloc, op.apply_Dbb_dag):
            fn(y, x, prec, nrhs)
            out.append(torch.empty_like(psi))
            op.unpack_half(out[-1], y, prec, nrhs)
        res.append((x.clone(), out))
    assert torch.equal(res[0][0], res[1][0])
    assert torch.equal(torch.view_as_real(res[0][1][0]), torch.view_as_real(res[1][1][0]))
    for a, b in zip(res[1][1][1:], res[0][1][1:]):
        assert _rel(a, b) <= tol

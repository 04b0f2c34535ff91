"""The sums of the CG by themselves: block sums into exact bins and into the sum tree, against
correctly rounded sums of the same numbers, and the first iterations of the fused CGs, whose
steps those sums decide, against the unfused ones."""
import ctypes
import importlib
import math
import os
import subprocess

import numpy as np
import pytest
import torch

from synthetic import gaussian_half5d, gaussian_source4d

from gpu_common import make_case

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "dwf_fields.cuh"
using namespace dwf;
__global__ void pairs(const float2* v, Reduce red) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  block_sum_pair(v[n], red, 0, gridDim.x, blockIdx.x);
}
__global__ void doubles(const double* v, Reduce red) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  block_sum_to(v[n], red, 0, gridDim.x, blockIdx.x);
}
__global__ void finish(SumIn in) { sum_in(in, 0, true); }
// one sum of blocks x threads numbers (FP32: slice pairs); work: zeros, at least
// kBins + blocks + 2 * groups + 3 words
extern "C" int run_sum(const void* v, int f64, int blocks, int threads, int use_bins, void* work, double* out) {
  Reduce r{};
  bin_t* bins = reinterpret_cast<bin_t*>(work);
  if (use_bins) {
    r.bins = bins;
  } else {
    const int groups = reduce_groups(blocks);
    r.partial = reinterpret_cast<double*>(work) + kBins;
    r.counter = reinterpret_cast<unsigned int*>(r.partial + blocks + groups);
    r.result = out;
    r.partial_stride = blocks + groups;
    r.counter_stride = groups + 1;
    r.result_stride = 1;
  }
  if (f64) doubles<<<blocks, threads>>>(reinterpret_cast<const double*>(v), r);
  else pairs<<<blocks, threads>>>(reinterpret_cast<const float2*>(v), r);
  if (use_bins) finish<<<1, 32>>>(SumIn{out, bins, 1});
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    build = importlib.import_module("paper_1501_04950_gb300.build")
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cu").write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", "-o", str(d / "sums.so"),
                                                              str(d / "sums.cu")], check=True)
    lib = ctypes.CDLL(str(d / "sums.so"))
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.run_sum.argtypes = [P, I, I, I, I, P, P]
    return lib


def _sum(lib, v, blocks, threads, bins):
    dev = torch.from_numpy(v).cuda()
    work = torch.zeros(72 + 2 * blocks + 64, dtype=torch.float64, device="cuda")
    out = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.run_sum(dev.data_ptr(), int(v.dtype == np.float64), blocks, threads, int(bins), work.data_ptr(),
                       out.data_ptr()) == 0
    return out.item()


def _numbers(kind, n, f64, seed):
    """Non-negative numbers as the squares of a field: alike, over the type's whole range, or a few
    large ones (more than 2^32 above the rest) among many small, zero and subnormal ones."""
    rng = np.random.default_rng(seed)
    if kind == "alike":
        v = rng.chisquare(24, n)
    elif kind == "range":
        v = 10.0 ** rng.uniform(-300 if f64 else -38, 300 if f64 else 36, n)
    else:
        v = rng.uniform(0, 1e-12, n)
        v[rng.integers(0, n, n // 4)] = 0.0
        v[rng.integers(0, n, 3)] = 5e-324 if f64 else 1e-44
        v[rng.integers(0, n, 2)] = 3e6
    return v.astype(np.float64 if f64 else np.float32)


@pytest.mark.parametrize("bins", [True, False])
@pytest.mark.parametrize("kind", ["alike", "range", "peaks"])
@pytest.mark.parametrize("f64,blocks,threads", [(0, 1, 32), (0, 7, 64), (0, 129, 128), (0, 300, 160), (1, 1, 32),
                                                (1, 129, 128), (1, 40, 256)])
def test_block_sums(lib, f64, blocks, threads, kind, bins):
    """FP32 pairs: exact but for summands cut at 2^-56 of the largest of their warp, once more per
    CTA: at most 2 * 2 * 160 * 2^-56 = 9e-15 of the sum.  FP64: a chain of at most 10 additions
    per CTA, 1.1e-16 each.  The tree adds at most 25 more.  Bins give the same value twice."""
    n = blocks * threads * (1 if f64 else 2)
    v = _numbers(kind, n, f64, blocks + threads)
    if threads == 160:   # the fifth warp, as the staged kernel's producer, adds zero
        v.reshape(blocks, threads, 2)[:, 128:] = 0.0
    ref = math.fsum(float(x) for x in v)
    got = _sum(lib, v, blocks, threads, bins)
    assert abs(got - ref) <= 9e-15 * ref
    assert got == _sum(lib, v, blocks, threads, bins)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("f64", [0, 1])
def test_sums_with_a_number_that_is_not_finite(lib, f64, bad):
    v = _numbers("alike", 3 * 128 * 2, f64, 1)
    v[257] = bad
    for bins in (True, False):
        assert not math.isfinite(_sum(lib, v, 3 if not f64 else 6, 128, bins))


def _op(sysm, **kw):
    from paper_1501_04950_gb300 import dwf
    op = dwf.DWF(sysm.lattice, sysm.Ls, sysm.M5, sysm.m, sysm.alpha, sysm.b, sysm.c,
                 bc_t=int(sysm.bc_t), rb_parity=sysm.black_parity, **kw)
    op.load_gauge(torch.from_numpy(sysm.U).cuda())
    return op


@pytest.mark.parametrize("L,Ls", [((4, 4, 2, 6), 8), ((4, 2, 6, 2), 10), ((8, 8, 8, 10), 16)])
@pytest.mark.parametrize("entry,prec,tol", [("cgne", 0, 1e-12), ("cgne", 1, 1e-5), ("cgne", 2, 1e-2),
                                            ("normal", 0, 1e-12), ("normal", 1, 1e-5)])
def test_first_iterations_match_the_unfused_cg(entry, prec, tol, L, Ls, monkeypatch):
    """The iterate after six steps (one poll), fused and unfused, on both sides of the direction
    split: its steps are quotients of the sums, so a sum that is off by e moves it by about e.
    Tolerances: the storage's rounding (1.1e-16, 6e-8, 4.9e-4) over some ten roundings a step."""
    from paper_1501_04950_gb300 import dwf
    sysm = make_case(L, Ls, "mobius", alpha=1.2, m=0.1, bc_t=-1)
    src = torch.from_numpy(gaussian_source4d(L, seed=1) if entry == "cgne" else gaussian_half5d(L, Ls, seed=2)).cuda()
    res = []
    for unfused in (False, True):
        if unfused:
            monkeypatch.setenv("DWF_UNFUSED_CG", "1")
        op = _op(sysm, precision_inner=prec, maxiter=6, check_every=6, reliable_delta=1e-6, rel_tol=1e-14)
        out = torch.zeros_like(src)
        if entry == "cgne":
            st = op.cgne_solve(src, out, allow_not_converged=True)[0]
            assert st["iterations"] == 6
        else:
            with pytest.raises(dwf.DWFError) as e:
                op.solve_normal(out, src)
            assert e.value.code == 4
        torch.cuda.synchronize()
        op.close()
        res.append(out)
    assert res[1].abs().max() > 0
    assert float(torch.linalg.norm(res[0] - res[1]) / torch.linalg.norm(res[1])) <= tol

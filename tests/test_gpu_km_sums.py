"""GPU: the tensor core's sums of the k-means distance passes against 64 bits.

The passes decide a point by bounds that charge a sum of P exact BF16 products
(P + 8) 2^-22 ||x|| ||c||: four times what rounding to nearest could lose, for
adders that truncate.  How the tensor core rounds is not documented, so its
error is measured here, on the passes' own kernels, with random operands and
such as lose most: many small products after a large one, products of one
sign, cancellation, and mantissas that are all ones."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def sums_lib(mr, tmp_path_factory):
    from paper_1309_0215_gb300 import _build
    out = str(tmp_path_factory.mktemp("km_sums"))
    flags = [*_build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", _build.INCLUDE, "--expt-relaxed-constexpr"]
    libs = {}
    jobs = []
    for name in ("km_tc_sums", "km_wide_sums"):
        libs[name] = os.path.join(out, name + ".so")
        jobs.append(subprocess.Popen([_build._nvcc(), *flags, "-shared", "-o", libs[name],
                                      os.path.join(HERE, "native", name + ".cu")]))
    assert [j.wait() for j in jobs] == [0, 0]
    tc, wide = ctypes.CDLL(libs["km_tc_sums"]), ctypes.CDLL(libs["km_wide_sums"])
    vp, u32 = ctypes.c_void_p, ctypes.c_uint32
    tc.km_tc_sums.argtypes = [vp, u32, u32, vp, u32, vp, vp, vp, ctypes.c_int]
    wide.km_wide_sums.argtypes = [vp, u32, u32, vp, u32, vp, vp, vp, vp]
    wide.km_wide_operands.argtypes = [u32, u32]
    wide.km_wide_operands.restype = ctypes.c_uint64
    return tc, wide


def _operands(kind, rows, d, rng, sign=1):
    """rows x d FP32 values; sign: of the last one of a row whose products cancel."""
    if kind == "normal":
        return rng.standard_normal((rows, d)).astype(np.float32)
    if kind == "positive":
        return rng.uniform(1, 2, (rows, d)).astype(np.float32)
    if kind == "ones in the mantissa":
        return np.full((rows, d), np.float32(2) - np.float32(2 ** -16)) * (1 + np.arange(rows)[:, None] % 7).astype(np.float32)
    if kind == "scales":
        return (rng.standard_normal((rows, d)) * 2.0 ** rng.integers(-14, 15, (rows, d))).astype(np.float32)
    # one large value somewhere, the others below the last bits of its products
    v = (rng.uniform(1, 2, (rows, d)) * 2.0 ** rng.integers(-13, -8, (rows, 1))).astype(np.float32)
    if kind == "large first":
        v[:, 0] = 1.9
    elif kind == "large anywhere":
        v[np.arange(rows), np.arange(rows) % d] = 1.9
    elif kind == "cancelled":
        v[:, 0], v[:, d - 1] = 1.9, sign * 1.9
    return v


KINDS = ["normal", "positive", "ones in the mantissa", "scales", "large first", "large anywhere", "cancelled"]


def _worst(got, x, c, products, terms):
    """The largest error in units of the charge."""
    import torch

    def split(a):
        t = torch.from_numpy(np.ascontiguousarray(a))
        hi = t.to(torch.bfloat16).float()
        return hi.double().numpy(), (t - hi).to(torch.bfloat16).double().numpy()

    (xh, xl), (ch, cl) = split(x), split(c)
    exact = xh @ ch.T
    if terms == 3:
        exact = exact + xh @ cl.T + xl @ ch.T
    norms = np.linalg.norm(x.astype(np.float64), axis=1)[:, None] * np.linalg.norm(c.astype(np.float64), axis=1)
    return float((np.abs(got - exact) / ((products + 8) * 2.0 ** -22 * norms)).max())


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("terms,d", [(3, 64), (3, 37), (1, 64)])
def test_tensor_core_sums_stay_within_their_charge(sums_lib, kind, terms, d):
    import torch
    rng = np.random.default_rng(d + terms)
    n, k = 3_000, 256
    x, c = _operands(kind, n, d, rng), _operands(kind, k, d, rng, -1)
    dx, dc = torch.from_numpy(x).cuda(), torch.from_numpy(c).cuda()
    zeros = torch.zeros(1024, device="cuda")
    work = torch.zeros(5 * n + 16, dtype=torch.int32, device="cuda")
    sums = torch.full(((n + 127) // 128 * 128, 256), float("nan"), device="cuda")
    torch.cuda.synchronize()
    assert sums_lib[0].km_tc_sums(dx.data_ptr(), n, d, dc.data_ptr(), k, zeros.data_ptr(), work.data_ptr(),
                                  sums.data_ptr(), terms) == 0
    torch.cuda.synchronize()
    assert not work[2:4].any()  # no wait gave up
    worst = _worst(sums[:n, :k].double().cpu().numpy(), x, c, 64 * terms, terms)
    print("worst error, of the charge:", worst)
    assert worst <= 1


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("d,k", [(256, 256), (128, 512), (70, 300), (20, 700)])
def test_wide_tensor_core_sums_stay_within_their_charge(sums_lib, kind, d, k):
    import torch
    rng = np.random.default_rng(d + k)
    n = 2_000
    x, c = _operands(kind, n, d, rng), _operands(kind, k, d, rng, -1)
    dx, dc = torch.from_numpy(x).cuda(), torch.from_numpy(c).cuda()
    zeros = torch.zeros(4096, device="cuda")
    bop = torch.zeros(sums_lib[1].km_wide_operands(d, k), dtype=torch.uint8, device="cuda")
    work = torch.zeros(5 * n + 16, dtype=torch.int32, device="cuda")
    chunks = (k + 255) // 256
    sums = torch.full(((n + 127) // 128 * 128, 256 * chunks), float("nan"), device="cuda")
    torch.cuda.synchronize()
    assert sums_lib[1].km_wide_sums(dx.data_ptr(), n, d, dc.data_ptr(), k, zeros.data_ptr(), bop.data_ptr(),
                                    work.data_ptr(), sums.data_ptr()) == 0
    torch.cuda.synchronize()
    assert not work[2:4].any()
    worst = _worst(sums[:n, :k].double().cpu().numpy(), x, c, 3 * 64 * ((d + 63) // 64), 3)
    print("worst error, of the charge:", worst)
    assert worst <= 1

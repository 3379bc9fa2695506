"""The all-pairs filter's contraction itself: for every pair of a tile the
tensor cores' result must be a lower bound of |y_i - y_j|^2, and its
accumulation may use no more than the share that the bound gives it.

The operands are the ones the product's epilogue writes (two FP16 terms per
component, the norms less the allowance, gemm_tc.cuh), formed here in numpy;
tests/filter_products.cu runs the MMAs of one 128 x 128 tile on them.  The
allowance restated (restructured.cu, op_bounds): kappa (s_i + s_j) + kabs with
kappa = 1.1 (5 2^-22 + (k + 2) 2^-24 + (steps + 4) 2^-21 + sqrt(k) 2^-25), of
which (steps + 4) 2^-21 stands for the accumulation, kabs = 1.1 (sqrt(k) + 1)
2^-24.  Rows at the largest norm (64), nearly equal rows (the sum cancels to a
millionth of its terms), components and norms over many magnitudes."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
f16, f32 = np.float16, np.float32


@pytest.fixture(scope="module")
def products(tmp_path_factory):
    torch = pytest.importorskip("torch")
    from paper_1807_03425_gb300 import build
    so = str(tmp_path_factory.mktemp("filter") / "filter_products.so")
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                   "-I" + build.CSRC, "-o", so, os.path.join(HERE, "filter_products.cu")], check=True)
    lib = ctypes.CDLL(so)

    def run(images, steps):
        d = torch.from_numpy(images).cuda()
        out = torch.zeros(128, 128, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        rc = lib.filter_products(ctypes.c_void_p(d.data_ptr()), steps, ctypes.c_void_p(out.data_ptr()),
                                 ctypes.c_void_p(status.data_ptr()))
        assert rc == 0 and int(status[0]) == 0
        return out.cpu().numpy().astype(np.float64)
    return run


def op_steps(k):
    return ((3 * ((k + 3) // 4) + 1) * 4 + 15) // 16


def allowance(k):
    kap = 5 * 2.0 ** -22 + (k + 2) * 2.0 ** -24 + (op_steps(k) + 4) * 2.0 ** -21 + np.sqrt(k) * 2.0 ** -25
    return f32(1.1 * kap), f32(1.1 * (np.sqrt(k) + 1) * 2.0 ** -24)


def operands(y):
    """A and B (128 x K FP16) and both images in core-matrix order."""
    k = y.shape[1]
    g, K = (k + 3) // 4, op_steps(k) * 16
    v = np.zeros((128, 4 * g), f32)
    v[:, :k] = y
    h = v.astype(f16)
    l = (v - h.astype(f32)).astype(f16)
    s = np.zeros(128, f32)
    for c in range(4 * g):
        s = (v[:, c].astype(np.float64) ** 2 + s).astype(f32)
    kap, kabs = allowance(k)
    sp = (s * (f32(1) - kap) - f32(0.5) * kabs).astype(f32)
    sh = sp.astype(f16)
    sl = (sp - sh.astype(f32)).astype(f16)
    A, B = np.zeros((128, K), f16), np.zeros((128, K), f16)
    for q in range(g):
        c, o = slice(4 * q, 4 * q + 4), 12 * q
        A[:, o:o + 4], A[:, o + 4:o + 8], A[:, o + 8:o + 12] = h[:, c], h[:, c], l[:, c]
        B[:, o:o + 4], B[:, o + 4:o + 8], B[:, o + 8:o + 12] = -2 * h[:, c], -2 * l[:, c], -2 * h[:, c]
    o = 12 * g
    A[:, o], A[:, o + 1], A[:, o + 2:o + 4] = sh, sl, 1
    B[:, o:o + 2], B[:, o + 2], B[:, o + 3] = 1, sh, sl

    def image(M):
        return M.reshape(16, 8, K // 8, 8).transpose(2, 0, 1, 3).copy().view(np.uint8).reshape(-1)
    return A, B, np.concatenate([image(A), image(B)])


def rows(k, seed):
    g = np.random.default_rng(seed)

    def to(y, r=63.9):
        return (y * (r / np.linalg.norm(y, axis=1, keepdims=True))).astype(f32)
    z, b = g.standard_normal((128, k)), np.abs(g.standard_normal((1, k)))
    yield to(z)
    yield to(np.abs(z))
    for e in (1e-1, 1e-2, 1e-3, 1e-4, 1e-6):
        yield to(b + e * z)
    yield to(np.abs(z) * 2.0 ** -np.arange(k) + 1e-3)
    yield to(np.abs(z) * 2.0 ** -np.arange(k)[::-1] + 1e-3)
    yield (to(np.abs(z)) * 2.0 ** -g.integers(0, 14, (128, 1))).astype(f32)
    yield (to(b + 1e-3 * z) * 2.0 ** -g.integers(0, 14, (128, 1))).astype(f32)
    yield (to(z) * 2.0 ** -10).astype(f32)
    yield to(z * 2.0 ** -g.integers(0, 16, (128, k)))


@pytest.mark.parametrize("k", [1, 5, 12, 16, 32])
def test_contraction_is_a_lower_bound(products, k):
    kap, kabs = (float(x) for x in allowance(k))
    for seed in range(8):
        for y in rows(k, 100 * k + seed):
            A, B, im = operands(y)
            out = products(im, op_steps(k))
            y = y.astype(np.float64)
            s = (y ** 2).sum(1)
            ss = s[:, None] + s[None]
            d2 = ((y[:, None, :] - y[None]) ** 2).sum(2)
            assert (out <= d2).all()
            assert (d2 - out <= 2 * (kap * ss + kabs)).all()  # and no looser than twice the allowance
            exact = A.astype(np.float64) @ B.astype(np.float64).T
            assert (np.abs(out - exact) <= (op_steps(k) + 4) * 2.0 ** -21 * ss).all()

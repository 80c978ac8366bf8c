"""The reciprocal and square root of the stage kernels (cpr_common.cuh:
frcp_ftz, fsqrt_ftz) against exact values and against CUDA's 1 / x and sqrt.

Bounds.  FP64: the hardware seeds carry 20 bits, a relative error d of at most
1.5 * 2^-20 with their truncation.  Reciprocal: the cut series leaves d^3 =
3e-18; square root: Newton's step leaves 1.5 d^2 and the residual correction,
with a factor good to d, 1.5 d^3 = 4.4e-18.  In units of the last place (at
least 2^-53 of the value) these are 0.03 and 0.04, the last operation rounds by
0.5: 0.55, and so never more than one unit from CUDA's rounded result.  FP32:
the instructions' documented bounds, one unit for the reciprocal and 2^-23
relative for the root, against exact values."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1709_01619_gb300 import build as b

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
TYPES = {"f32": (np.float32, torch.float32), "f64": (np.float64, torch.float64)}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("native_math") / "native_math.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-shared", os.path.join(HERE, "native_math.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


def evaluate(lib, kind, x):
    nt, tt = TYPES[kind]
    d = torch.tensor(np.asarray(x, dtype=nt), device="cuda")
    out = [torch.empty_like(d) for _ in range(4)]
    torch.cuda.synchronize()
    f = getattr(lib, f"native_math_{kind}")
    assert f(*[ctypes.c_void_p(t.data_ptr()) for t in (d, *out)], ctypes.c_int(d.numel())) == 0
    return [t.cpu().numpy() for t in out]


def units(got, exact):
    """Distance in units of the last place of the rounded exact value."""
    r = np.abs(exact).astype(got.dtype)
    return np.abs(got - exact) / (np.nextafter(r, got.dtype.type(np.inf)) - r).astype(exact.dtype)


def samples(kind, lo, hi):
    """Mantissas over a grid and at random, exponents lo..hi."""
    rng = np.random.default_rng(5)
    m = np.concatenate([1.0 + np.arange(4096) / 4096.0, 1.0 + rng.random(60000), 2.0 - 2.0 ** -np.arange(1, 24)])
    return np.ldexp(m, rng.integers(lo, hi + 1, m.size)).astype(TYPES[kind][0])


def test_fp64_rounds_within_0_55_units(lib):
    x = samples("f64", -960, 1020)
    r, s, r0, s0 = evaluate(lib, "f64", x)
    wide = x.astype(np.longdouble)
    assert units(r, 1 / wide).max() <= 0.55
    assert units(s, np.sqrt(wide)).max() <= 0.55
    assert np.abs(r.view(np.int64) - r0.view(np.int64)).max() <= 1
    assert np.abs(s.view(np.int64) - s0.view(np.int64)).max() <= 1


def test_fp32_within_the_instructions_bounds(lib):
    x = samples("f32", -125, 125)
    r, s, _, _ = evaluate(lib, "f32", x)
    wide = x.astype(np.float64)
    assert units(r, 1 / wide).max() <= 1.0
    assert (np.abs(s - np.sqrt(wide)) <= 2.0 ** -23 * np.sqrt(wide)).all()


@pytest.mark.parametrize("kind", ["f32", "f64"])
def test_special_operands(lib, kind):
    """Zeros, infinities, NaN and negative operands as IEEE; subnormal operands
    count as zeros, results below the normal range come out as zeros (the root
    of a subnormal FP64 operand as the operand, below 1e-307 either way)."""
    nt = TYPES[kind][0]
    tiny = np.finfo(nt).tiny
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, -np.finfo(nt).max, tiny, 1.0], dtype=nt)
    r, s, r0, s0 = evaluate(lib, kind, x)
    np.testing.assert_array_equal(s[:7], s0[:7])
    np.testing.assert_array_equal(np.signbit(s[:2]), np.signbit(s0[:2]))
    np.testing.assert_array_equal(r[:5], r0[:5])
    np.testing.assert_array_equal(np.signbit(r[:4]), np.signbit(r0[:4]))
    np.testing.assert_allclose([r[7], r[8], s[7], s[8]], [r0[7], r0[8], s0[7], s0[8]], rtol=2 * np.finfo(nt).eps)
    sub = np.array([tiny / 2, tiny / 1024, -tiny / 2], dtype=nt)
    r, s, _, _ = evaluate(lib, kind, sub)
    np.testing.assert_array_equal(r, [np.inf, np.inf, -np.inf])
    assert (s[:2] >= 0).all() and (s[:2] <= tiny).all()
    assert np.isnan(s[2]) or s[2] == 0
    big = np.array([np.finfo(nt).max, -np.finfo(nt).max], dtype=nt)
    r, _, _, _ = evaluate(lib, kind, big)
    np.testing.assert_array_equal(r, [0.0, -0.0])

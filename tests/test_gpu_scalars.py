"""The scalar routines that stand in for FP64 instructions, against those instructions:
rcp64 and rsqrt64 (reciprocal and root from FP32 starts), cut_f32 and
widen_f64 (conversions on the integer pipe), df_to_f64 (the double nearest to a
double-float).

Tolerances, from the roundings each makes: rcp64 rounds once, at the end, of a value good
to 2^-64: half an ulp and 1e-3 of one. rsqrt64 rounds x r (2^-53, halved by the
series) and its result: 1.5 * 2^-53 and 1e-3 of it. The conversions are exact."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build
    out = str(tmp_path_factory.mktemp("scalars") / "libscalars.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS +
                   ["-shared", "-o", out, os.path.join(HERE, "device_scalars.cu")], check=True, capture_output=True)
    return ctypes.CDLL(out)


def _run(fn, inputs, outputs):
    """fn(n, device copies of the inputs, device outputs of the given types) as numpy arrays."""
    import torch
    dev = [torch.tensor(v, device="cuda") for v in inputs]
    out = [torch.empty(len(inputs[0]), dtype=t, device="cuda") for t in outputs]
    assert fn(len(inputs[0]), *[ctypes.c_void_p(t.data_ptr()) for t in dev + out]) == 0
    return [t.cpu().numpy() for t in out]


def _ulps(got, want):
    """Error of got in ulps of the long double value want."""
    return np.abs(got.astype(np.longdouble) - want) / np.spacing(np.abs(got)).astype(np.longdouble)


def test_reciprocal_root_and_conversions(lib):
    import torch
    rng = np.random.default_rng(11)
    n = 1 << 20
    mant = rng.uniform(1, 2, n)
    mant[:64] = 1 + np.arange(64) * 2.0 ** -52      # at the binade's lower edge
    mant[64:128] = 2 - (1 + np.arange(64)) * 2.0 ** -52  # at its upper edge
    b = np.ldexp(mant, rng.integers(-160, 160, n)) * rng.choice([-1.0, 1.0], n)  # in and out of FP32's range
    f8, f4 = torch.float64, torch.float32
    rcp, div, rsq, cut, wide = _run(lib.scalars_f64, [b], [f8, f8, f8, f4, f8])
    B = b.astype(np.longdouble)
    assert np.max(_ulps(rcp, 1 / B)) <= 0.501
    assert np.max(np.abs(rcp - div) / np.spacing(np.abs(div))) <= 1 and np.mean(rcp == div) > 0.999
    r = rsq.astype(np.longdouble)
    assert np.max(np.abs(1 - np.abs(B) * r * r)) / 2 <= 1.5 * 2.0 ** -53 * (1 + 1e-3)
    # cut towards zero, flushed below FP32's normal range
    with np.errstate(over="ignore", under="ignore"):
        near = b.astype(np.float32)
    down = np.where(np.abs(near.astype(np.float64)) > np.abs(b), np.nextafter(near, np.float32(0)), near)
    tiny, huge = np.abs(b) < 2.0 ** -126, np.abs(b) >= 2.0 ** 128
    assert np.array_equal(cut[~tiny & ~huge], down[~tiny & ~huge])
    assert np.all(cut[tiny] == 0) and np.all(np.isinf(cut[huge]))
    ok = (np.abs(near) >= np.float32(2.0 ** -126)) & np.isfinite(near)
    assert np.array_equal(wide[ok], near[ok].astype(np.float64))
    assert np.all(wide[np.abs(near) < np.float32(2.0 ** -126)] == 0)


def test_double_float_to_double(lib):
    import torch
    rng = np.random.default_rng(5)
    n = 1 << 20
    hi = np.ldexp(rng.uniform(1, 2, n), rng.integers(-80, 100, n)).astype(np.float32)  # both sides of 2^-70
    hi[: n // 4] = np.ldexp(1.0, rng.integers(-80, 100, n // 4)).astype(np.float32)     # powers of two
    hi[n // 4: n // 2] = np.nextafter(np.ldexp(2.0, rng.integers(-80, 100, n // 4)).astype(np.float32), np.float32(0))
    hi *= rng.choice(np.array([-1, 1], dtype=np.float32), n)
    half = np.spacing(np.abs(hi)) / 2
    lo = (half * rng.uniform(-1, 1, n)).astype(np.float32)
    k = rng.integers(0, n, n // 8)
    lo[k] = half[k] * rng.choice(np.array([-1, 1], dtype=np.float32), n // 8)  # half an ulp of hi
    k = rng.integers(0, n, n // 8)  # ties of the result's own rounding
    lo[k] = (half[k] * (2.0 ** -29 * (2 * rng.integers(-2 ** 20, 2 ** 20, n // 8) + 1))).astype(np.float32)
    lo[rng.integers(0, n, n // 8)] = 0
    hi = np.concatenate([hi, np.array([0, -0.0, 1e-45, -1e-40, np.inf, -np.inf, np.nan, 3.4e38], dtype=np.float32)])
    lo = np.concatenate([lo, np.array([0, 0, 0, 0, 0, 0, 0, 1e30], dtype=np.float32)])
    got, want = _run(lib.scalars_df, [hi, lo], [torch.float64, torch.float64])
    assert np.array_equal(got, want, equal_nan=True)

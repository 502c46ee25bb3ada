"""The prompt GEMM's silu divides by an approximate reciprocal and adds the quotient's remainder: its bound of 0.51 units in
the last place, for every reciprocal within the two units that CUDA documents for the fast division.  (The arithmetic alone, in
numpy; test_gpu_silu.py runs the device function.)"""
import numpy as np


def test_corrected_quotient_is_within_its_bound():
    rng = np.random.default_rng(0)
    n = 1 << 20
    x = (rng.standard_normal(n) * np.exp(rng.uniform(-10, 4, n))).astype(np.float32)
    d = (1 + np.exp(rng.uniform(-20, 80, n))).astype(np.float32)
    r = (1 / d.astype(np.float64)).astype(np.float32)
    r = (r + rng.integers(-2, 3, n) * np.spacing(r)).astype(np.float32)
    q = x * r
    x64, d64, q64, r64 = (v.astype(np.float64) for v in (x, d, q, r))
    rem = (x64 - q64 * d64).astype(np.float32)                       # exact products in double: one rounding, as a fused step
    z = (q64 + rem.astype(np.float64) * r64).astype(np.float32)
    exact = x.astype(np.longdouble) / d.astype(np.longdouble)
    normal = np.abs(exact) > 1e-36
    assert (np.abs(z - exact) / np.spacing(np.abs(z)))[normal].max() < 0.51

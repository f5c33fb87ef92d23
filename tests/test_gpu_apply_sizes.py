"""The FP32 LS-apply at the edges of its transform lengths, against the oracle.

The padded length P is the smallest power of two >= 2 n - 1 (Sec. 2); lengths 32 to 4096 have
their own kernels, chained by programmatic launches, one or several transforms per CTA.
Checked: both sides of every change of P up to 1024, applied twice in a row in place (a call
starts while the one before it may still run), with every column-tile shape the length has.
Bound: FP32 FFT rounding, a few log2(P) ulps (2^-24) normwise, with a factor of 10.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import greens  # noqa: E402
from paper_1602_07652_gb300 import binding, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1602_07652_gb300 import build_lib
    build_lib.build()
    binding.load()


@pytest.mark.parametrize("n", [8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256, 258, 512])
def test_fp32_apply_at_the_edges_of_each_length(n):
    w = inputs.omega_for_ppw(n, 10.24)
    m = inputs.bump_medium(n, nbumps=5, seed=n)
    L = next(d for d in range(1, n + 1) if n % d == 0 and n // d + 4 <= 112)
    s = binding.Solver(torch.from_numpy(m), w, layers=L, ext=2, precision=binding.LS_MIXED)
    u = inputs.random_field(n, n)
    once = greens.apply_H(u, m, 1.0 / n, w)
    ref = greens.apply_H(once, m, 1.0 / n, w)
    tol = 10 * 2 * 2 * math.log2(2 * n) * 2.0 ** -24
    for shape in (None, 0, 1, 2, 3, 4, 5, 6, 7, 8):
        if shape is not None:
            s.ls_set_shapes(shape)
        y = torch.from_numpy(u.astype(np.complex64)).cuda()
        s.ls_apply_f32(y, y)
        s.ls_apply_f32(y, y)
        err = np.linalg.norm(y.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err < tol, (shape, err)
    s.close()


@pytest.mark.parametrize("n", [16, 17, 32, 33, 63, 64, 65, 129, 256, 257, 513])
def test_fp64_and_double_float_applies_at_the_edges_of_each_length(n):
    # P = 64 .. 2048 have kernels of their own (P = 32: the generic ones); two applies in a
    # row in place, and the incident right-hand side.  Bounds: FP64 FFT rounding and the
    # double-float format's 2^-46 against the FP64 result, with a factor of 10 each; the
    # kernel weights' own rounding against the oracle.
    w = inputs.omega_for_ppw(n, 10.24)
    m = inputs.bump_medium(n, nbumps=5, seed=n)
    L = next(d for d in range(1, n + 1) if n % d == 0 and n // d + 4 <= 112)
    s = binding.Solver(torch.from_numpy(m), w, layers=L, ext=2, precision=binding.LS_MIXED)
    u = inputs.random_field(n, n)
    ref = greens.apply_H(greens.apply_H(u, m, 1.0 / n, w), m, 1.0 / n, w)
    out = {}
    for name, fn in (("fp64", s.ls_apply), ("df", s.ls_apply_double_float)):
        y = torch.from_numpy(u).cuda()
        fn(y, y)
        fn(y, y)
        out[name] = y.cpu().numpy()
        assert np.linalg.norm(out[name] - ref) / np.linalg.norm(ref) < 1e-11, name
    assert np.linalg.norm(out["df"] - out["fp64"]) / np.linalg.norm(ref) < 10 * 2 * math.log2(2 * n) * 2.0 ** -46
    f = greens.rhs(m, 1.0 / n, w, greens.incident_plane_wave(n, w, 0.3))
    for df in (1, 0):
        s.ls_set_double_float(df)
        g = s.ls_incident_rhs(0.3).cpu().numpy()
        assert np.linalg.norm(g - f) / np.linalg.norm(f) < 1e-11, df
    s.close()

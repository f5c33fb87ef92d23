"""Kernels launched programmatically read what their predecessor writes with ordinary loads.

Such a kernel is resident while its predecessor still runs (ls_internal.cuh, pdl_wait).  The
read-only path (__ldg, ldg_c, const __restrict__ parameters) is for memory that nothing writes
while a kernel is resident, so in these kernels it may serve constants only: factors, coupling
tables, twiddles and the kernel's spectrum, all written before the handle is returned.  The
first tests check that in the sources; the last runs chains on a GPU.
"""
import math
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1602_07652_gb300", "csrc")

# what a chained kernel may read through the read-only path: parameters by name, and loads by
# the expression they address
CONST_PARAMS = {"tw", "ghat"}
CONST_LOADS = [r"tw\[", r"g\[", r"Ms\[", r"w < 3 \* q \? &a\.cp\.cw\[", r"wi\[", r"ei\["]


def _sources():
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            out[f] = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
    return out


def _braced(text, at):
    """text from the first brace at or after at to its partner"""
    i = text.index("{", at)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def _chained_kernels():
    for f, text in _sources().items():
        for k in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)\s*)?"
                             r"(\w+)\s*\(((?:[^()]|\([^()]*\))*)\)\s*\{", text):
            body = _braced(text, k.end() - 1)
            if "pdl_wait()" in body or "griddepcontrol.wait" in body:
                yield f, k.group(1), k.group(2), body


def test_the_chained_kernels_are_found():
    names = {name for _, name, _, _ in _chained_kernels()}
    assert names == {"k_rows16_fwd", "k_cols16", "k_cols16_tma", "k_cols16_tma2", "k_rows16_inv", "k_wide_rows_fwd",
                     "k_wide_cols", "k_wide_rows_inv", "k_cr_step", "k_cr_even", "k_cr_mma", "k_dense_mma"}


def test_chained_kernels_take_only_constants_as_read_only():
    for f, name, params, body in _chained_kernels():
        for p in re.split(r",(?![^<]*>)", params):
            if re.search(r"\bconst\b", p) and "__restrict__" in p:
                assert p.split()[-1].lstrip("*&") in CONST_PARAMS, (f, name, p.strip())
        for load in re.finditer(r"(?:__ldg|ldg_c)\(&?([^;]*)", body):
            assert any(re.match(c, load.group(1)) for c in CONST_LOADS), (f, name, load.group(0))


def test_sources_and_sinks_of_chained_kernels_use_ordinary_loads():
    seen = set()
    for f, text in _sources().items():
        for s in re.finditer(r"struct (SrcMU|SrcInc|SrcIncDf|DstApply|DstRhs|RhsSrc)\s*\{", text):
            seen.add(s.group(1))
            body = _braced(text, s.end() - 1)
            assert not re.search(r"__ldg|ldg_c|__restrict__", body), (f, s.group(1))
    assert seen == {"SrcMU", "SrcInc", "SrcIncDf", "DstApply", "DstRhs", "RhsSrc"}


@pytest.mark.gpu
@pytest.mark.parametrize("n", [33, 65, 127, 255, 301, 513, 801])
def test_chained_calls_equal_calls_that_wait(n):
    # in place, so that each call reads what the one before it writes; the arithmetic of a call
    # is fixed, so the results are the same bits
    torch = pytest.importorskip("torch")
    from paper_1602_07652_gb300 import binding, build_lib, inputs
    build_lib.build()
    L = next(d for d in range(1, n + 1) if n % d == 0 and n // d + 4 <= 112)
    m = torch.from_numpy(inputs.bump_medium(n, nbumps=5, seed=n))
    s = binding.Solver(m, inputs.omega_for_ppw(n, 10.24), layers=L, ext=2, precision=binding.LS_MIXED)
    u = torch.from_numpy(inputs.random_field(n, n)).cuda()
    u /= math.sqrt(float(np.vdot(u.cpu().numpy(), u.cpu().numpy()).real))

    def chain(fn, dtype, wait):
        y = u.to(dtype, copy=True)
        for _ in range(6):
            fn(y, y)
            if wait:
                torch.cuda.synchronize()
        return y.cpu()

    shapes = [None, 0, 2, 3, 4, 5, 6, 7, 8] if 2 * n - 1 > 128 else [None]   # P >= 256
    for shape in shapes:
        if shape is not None:
            s.ls_set_shapes(shape)
        ref = chain(s.ls_apply_f32, torch.complex64, True)
        for _ in range(5):
            assert torch.equal(chain(s.ls_apply_f32, torch.complex64, False), ref), shape
    for fn in (s.ls_apply, s.ls_apply_double_float):
        ref = chain(fn, torch.complex128, True)
        for _ in range(5):
            assert torch.equal(chain(fn, torch.complex128, False), ref), fn.__name__
    for df in (1, 0):   # the incident wave's factors are written by the kernel before the row pass
        s.ls_set_double_float(df)
        ref = []
        for k in range(6):
            ref.append(s.ls_incident_rhs(0.3 + k))
            torch.cuda.synchronize()
        got = [s.ls_incident_rhs(0.3 + k) for k in range(6)]
        assert all(torch.equal(a, b) for a, b in zip(got, ref)), df
    s.close()

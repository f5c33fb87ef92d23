"""Shared-memory limits of the kernels hold for every handle of the process.

The limit (dynamic shared memory beyond 48 KB) belongs to a kernel, not to a handle: whatever
other handles there are, and whichever thread made them, a handle's calls must launch.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1602_07652_gb300 import binding, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1602_07652_gb300 import build_lib
    build_lib.build()
    binding.load()


def solver(n, layers, ext, prec=None, **kw):
    m = torch.from_numpy(inputs.bump_medium(n, nbumps=4, seed=n)).cuda()
    return binding.Solver(m, inputs.omega_for_ppw(n, 10.0), layers=layers, ext=ext,
                          precision=binding.LS_MIXED if prec is None else prec, **kw)


def test_a_failed_or_finished_autotune_leaves_a_shape_that_works():
    # n = 1025: P = 4096, whose generic column pass needs 144 KB; n = 520: P = 2048, 72 KB
    s = solver(1025, 25, 10)
    u = torch.from_numpy(inputs.random_field(1025, 1).astype(np.complex64)).cuda()
    ref = s.ls_apply_f32(u)
    o = solver(520, 10, 10)
    try:
        s.ls_autotune(1, 1)
    except RuntimeError:
        pass
    y = s.ls_apply_f32(u)
    assert float((y - ref).abs().square().sum() / ref.abs().square().sum()) < 1e-10
    o.close()
    s.close()


def test_a_handle_of_a_shorter_transform_leaves_a_longer_one_its_shared_memory():
    s = solver(1025, 25, 10)
    u = torch.from_numpy(inputs.random_field(1025, 1).astype(np.complex64)).cuda()
    ref = s.ls_apply_f32(u)
    s.ls_set_shapes(1)   # the generic passes

    def check():
        y = s.ls_apply_f32(u)
        assert float((y - ref).abs().square().sum() / ref.abs().square().sum()) < 1e-10

    check()
    k = solver(64, 2, 6)   # the first call without allocation sets a limit of its own
    g = k.ls_get_spectrum()[0].to(torch.complex64).contiguous()
    m = torch.zeros((64, 64), dtype=torch.float32, device="cuda")
    binding.ls_apply_f32_noalloc(64, m, g, torch.zeros((64, 64), dtype=torch.complex64, device="cuda"))
    check()
    o = solver(520, 10, 10)
    check()
    s.ls_autotune(1, 1)
    for x in (k, o, s):
        x.close()


def test_factorisations_of_different_heights_in_several_threads():
    # q = 112 needs 204 KB a CTA for the inverses, q = 54 needs 51 KB
    tall = solver(400, 4, 6, binding.LS_FP64, stream=torch.cuda.Stream())
    short = [solver(50, 1, 2, binding.LS_FP64, stream=torch.cuda.Stream()) for _ in range(4)]
    torch.cuda.synchronize()
    errors, done = [], threading.Event()

    def factor(s, more):
        try:
            while more():
                s.ls_factor()
        except RuntimeError as e:
            errors.append(e)

    others = [threading.Thread(target=factor, args=(s, lambda: not done.is_set())) for s in short]
    for t in others:
        t.start()
    left = iter(range(10))
    factor(tall, lambda: next(left, None) is not None)
    done.set()
    for t in others:
        t.join()
    assert not errors, errors
    for s in short + [tall]:
        s.close()


def test_a_taller_strip_is_factored_after_a_handle_of_a_shorter_one():
    # the steps that build the reduced inverse ask for 60 KB at q = 112, 50 KB at q = 70
    tall = solver(200, 2, 6, binding.LS_FP64)
    short = solver(100, 2, 10, binding.LS_FP64)
    tall.ls_factor()
    short.close()
    tall.close()

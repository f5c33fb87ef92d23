"""Block-cyclic-reduction steps on the CUDA cores at the sizes where their splitting can go wrong.

The local solves (C^l)^{-1} b (Sec. 3.4; factors of Sec. 4.1) run one launch per level, the
blocks of a level cut into chunks of rows, the odd blocks' D^{-1} b taken on the forward way and
the last levels replaced by the inverse of their reduced system.  Checked against the oracle's
banded-LU solve: few and odd numbers of blocks (the inverse starts at the second level or
later), strip heights that the chunks do not divide, one and several chunks, every batch form;
and Algorithm 2's sweeps with their injections against the oracle's.  Bounds: those of the
other local-solve tests (FP32 rounding in mixed precision, the conditioning of the strips in FP64).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import polarized, sparsify  # noqa: E402
from paper_1602_07652_gb300 import binding, inputs  # noqa: E402

# n blocks, L layers, E: q = n / L + 2 E = 9, 15, 24, 45, 57, 104
SIZES = [(10, 2, 2), (9, 1, 3), (24, 3, 8), (37, 1, 4), (111, 3, 10), (168, 2, 10)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1602_07652_gb300 import build_lib
    build_lib.build()
    binding.load()


@pytest.mark.parametrize("prec,tol", [(binding.LS_FP64, 1e-7), (binding.LS_MIXED, 2e-4)])
@pytest.mark.parametrize("n,L,E", SIZES)
def test_local_solves_and_batches_match_oracle(n, L, E, prec, tol):
    w = inputs.omega_for_ppw(n, 10.0)
    m = inputs.bump_medium(n, nbumps=4, seed=n)
    s = binding.Solver(cuda(m), w, layers=L, ext=E, precision=prec)
    s.ls_factor()
    if prec == binding.LS_MIXED:
        s.ls_set_tensor_steps(0)
    st = sparsify.Stencils(n, 1.0 / n, w)
    lays = (polarized.Layering(m, st, w, L, E), polarized.Layering(m.T.copy(), st.transposed(), w, L, E))
    bd = polarized.BiDirectional(m, st, w, L, E)
    g = np.stack([inputs.random_field(n, 60 + b) for b in range(8 if prec == binding.LS_MIXED else 4)])
    for split in (1, 0):
        s.ls_set_reduction(split)
        for d in (0, 1):
            for l in sorted({0, L - 1}):
                b = inputs.random_field(n, 7 * l + d, nz=lays[d].q)
                assert rel(s.ls_local_solve(d, l, cuda(b)).cpu().numpy(), lays[d].solve_local(l, b)) < tol, (split, d, l)
        for nb in (1, 2, 3, 4, 8):
            if nb <= len(g):
                v = s.ls_precond_bd_batch(cuda(g[:nb])).cpu().numpy()
                for b in range(nb):
                    assert rel(v[b], bd(g[b])) < tol, (split, nb, b)
    s.close()


def test_a_handle_of_shorter_strips_leaves_a_taller_one_its_shared_memory():
    # q = 112, then handles of q = 104 and 100 on the same kernels: in batches of 8 all ask for
    # more than 48 KB a CTA, the first for the most
    n = 200
    w = inputs.omega_for_ppw(n, 10.0)
    m = cuda(inputs.bump_medium(n, nbumps=4, seed=3))
    s = binding.Solver(m, w, layers=2, ext=6, precision=binding.LS_MIXED)
    s.ls_factor()
    s.ls_set_tensor_steps(0)
    g = cuda(np.stack([inputs.random_field(n, 70 + b) for b in range(8)]))
    alone = s.ls_precond_bd_batch(g).cpu()
    others = [binding.Solver(m, w, layers=2, ext=2, precision=binding.LS_MIXED),
              binding.Solver(m[:180, :180].contiguous(), w, layers=2, ext=5, precision=binding.LS_MIXED)]
    assert torch.equal(s.ls_precond_bd_batch(g).cpu(), alone)
    for o in others + [s]:
        o.close()

"""Kernels and dispatch rules at the sizes where they can go wrong, each against the oracle or
the general path: window edges of the Q1 mass solve."""
import numpy as np
import pytest

import oracle as O
import synth_inputs as S
from conftest import check_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda").contiguous()


@pytest.mark.parametrize("n,leaf_max,nrhs", [(8, 16, 1), (16, 16, 3), (32, 64, 2), (64, 64, 1), (128, 64, 5)])
def test_q1_mass_solve_windows(n, leaf_max, nrhs):
    # the mass solve runs windows of 64 nodes with a 32-node halo: grids below one window, one
    # window, several, and line counts that do not fill a block.  The solution does not depend
    # on the preconditioner, the count of PCG does: no more than the oracle's plus one.
    from paper_1308_3339_gb300 import FmmPreconditioner
    h = 1.0 / (n + 1)
    f = np.stack([S.gaussian_mixture(n, 40 + r) for r in range(nrhs)])
    P = FmmPreconditioner(n, p=10, leaf_max=leaf_max, precision="fp64", n_rhs=nrhs)
    P.set_operator("q1")
    u, info = P.solve(dev(f), method="cg", rtol=1e-10)
    R = O.Problem(n, p=10, leaf_max=leaf_max)
    R.set_operator("q1")
    counts = []
    for r in range(nrhs):
        uo, it, _, _ = R.solve(O.q1_load(n, h, f[r]), "cg", 30, 200, 1e-10, "fmm")
        counts.append(it)
        check_close(f"q1 windows n={n} rhs={r}", u[r].cpu().numpy().ravel(), uo, 1e-8, 1e-8)
    assert info["iters"] <= max(counts) + 1, (info["iters"], counts)
    P.close()

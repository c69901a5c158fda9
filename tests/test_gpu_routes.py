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


@pytest.mark.parametrize("n,leaf_max,prec,nrhs", [(32, 16, "fp64", 2), (64, 256, "fp32", 3), (128, 64, "mixed_tf32", 1),
                                                  (128, 16, "fp32", 1)])
def test_first_apply_bc_under_capture_sums_directly(n, leaf_max, prec, nrhs):
    # a first apply_bc inside a stream capture cannot form its tables and sums the boundary data
    # directly; later calls take the tables.  Same operator either way: FP64 to its rounding,
    # single precision to FP32 sums of ~100 terms (1e-5).
    from paper_1308_3339_gb300 import FmmPreconditioner
    f = dev(np.stack([S.gaussian_mixture(n, 60 + r) for r in range(nrhs)]))
    g = dev(np.stack([S.random_field(n, 70 + r)[: 4 * n] for r in range(nrhs)]))
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        P = FmmPreconditioner(n, p=10, leaf_max=leaf_max, precision=prec, n_rhs=nrhs, stream=st)
        u = torch.empty_like(f)
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            P.apply_bc(f, g, out=u)
        graph.replay()
        st.synchronize()
        ut = P.apply_bc(f, g)
        st.synchronize()
    tol = 1e-12 if prec == "fp64" else 1e-5
    check_close(f"apply_bc direct vs tables {prec} n={n}", ut.cpu().numpy(), u.cpu().numpy(), tol, tol)
    P.close()

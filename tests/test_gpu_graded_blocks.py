"""Stack blocks whose columns differ by orders of magnitude.

Free fermions (U = g = 0): e^{V} = 1, and on the eigenvectors of K the slices
multiply column k by e^{-dtau eps_k}, so that within a block of n slices the
columns grow apart by up to e^{3 n dtau}.  The QR factors do not see the
columns' scale, so the weight stays accurate at any grading as long as the
products and the Gram matrix keep every column's own digits.  The weight is
log|det P^T e^{-2 Theta K} P|, evaluated here through the eigenvalues of K."""
import numpy as np
import pytest

from oracle import pqmc as opq
from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda():
    import torch
    torch.cuda.set_device(0)
    pqmc.load()


def free(L, dtau):
    """The chain and its exact log weight per spin (the trial's symmetry breaking included)."""
    spec = workloads.honeycomb(L, U=0.0, dtau=dtau, two_theta=20 * dtau, g=0.0, M_N=0.0)
    m = opq.Model(opq.Params(kind=spec.kind, Lx=L, Ly=L, U=0.0, dtau=dtau, two_theta=spec.two_theta, g=0.0, M_N=0.0, n_stab=10))
    w, V = np.linalg.eigh(m.K)
    exact = []
    for sg in (1, -1):
        A = m.P[sg].T @ V
        exact.append(np.linalg.slogdet((A * np.exp(-spec.two_theta * (w - w[0]))) @ A.T)[1] - m.P[sg].shape[1] * spec.two_theta * w[0])
    return spec, exact


# A log weight is a sum of N/2 logarithms per block with FP64 errors, some 1e-16 each relative to the
# total: 1e-14 of it, times 10.
@pytest.mark.parametrize("L,dtau", [(3, 0.5), (6, 0.1), (6, 0.5), (6, 0.8)])
def test_weight_of_graded_blocks_fp64(L, dtau):
    spec, exact = free(L, dtau)
    for tpb in (64, 128, 256):
        ctx = pqmc.Context([spec], prec=pqmc.FP64, seed=1, n_stab=10, cta_threads=tpb)
        w = ctx.weight()
        assert abs(w[0] - exact[0]) < 1e-13 * abs(exact[0]) + 1e-13 and abs(w[2] - exact[1]) < 1e-13 * abs(exact[1]) + 1e-13, (w, exact)
        ctx.close()


@pytest.mark.parametrize("L,dtau", [(3, 0.5), (6, 0.1), (6, 0.8), (9, 0.5)])
def test_weight_of_graded_blocks_spread(L, dtau):
    """The same by the whole-GPU sweep, whose factor comes from the Gram matrix."""
    spec, exact = free(L, dtau)
    ctx = pqmc.Context([spec], prec=pqmc.FP64, seed=1, n_stab=10, spread=1)
    w = ctx.weight()
    assert abs(w[0] - exact[0]) < 1e-13 * abs(exact[0]) + 1e-13 and abs(w[2] - exact[1]) < 1e-13 * abs(exact[1]) + 1e-13, (w, exact)
    ctx.close()

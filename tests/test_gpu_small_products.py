"""The stabilisation's FP64 products by FMAs (up to 16 orbitals) and by digits
(from 17 on), on both sides of the line and below it, with equal and unequal
spins: G at every stabilisation point and the weight of given fields against
the oracle, to the 1e-4 of the FP32 path (weights, a sum of 2 Ltau / n_stab logarithms of
FP32 blocks: 1e-5 relative)."""
import numpy as np
import pytest

from oracle import pqmc as opq
from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,Lx,Ly,n_up,n_dn", [
    (workloads.HONEYCOMB, 2, 2, 4, 4), (workloads.HONEYCOMB, 3, 3, 9, 9), (workloads.HONEYCOMB, 3, 3, 1, 9),
    (workloads.HONEYCOMB, 4, 4, 16, 16), (workloads.SQUARE, 5, 5, 12, 11), (workloads.SQUARE, 6, 6, 16, 13),
    (workloads.SQUARE, 6, 6, 17, 16), (workloads.SQUARE, 6, 6, 17, 17)])
@pytest.mark.parametrize("tpb,dense", [(64, 0), (256, 0), (64, 1)])
def test_green_and_weight(kind, Lx, Ly, n_up, n_dn, tpb, dense):
    import torch
    torch.cuda.set_device(0)
    spec = workloads.ChainSpec(kind=kind, Lx=Lx, Ly=Ly, tp=-0.2 if kind == workloads.SQUARE else 0.0, U=4.0, two_theta=2.0,
                               g=0.3, M_N=0.21, n_up=n_up, n_dn=n_dn)
    fields = workloads.random_fields(spec, seed=5)
    m = opq.Model(opq.Params(kind=kind, Lx=Lx, Ly=Ly, tp=spec.tp, U=spec.U, dtau=spec.dtau, two_theta=spec.two_theta, g=spec.g,
                             M_N=spec.M_N, n_up=n_up, n_dn=n_dn, n_stab=2))
    ctx = pqmc.Context([spec], prec=pqmc.FP32, seed=5, n_stab=2, cta_threads=tpb, dense_chains=dense)
    ref = pqmc.Context([spec], prec=pqmc.FP64, seed=5, n_stab=2)
    for c in (ctx, ref):
        c.set_fields(fields)
    for b in (0, 3, m.Ltau // 2):
        for s, sg in ((0, 1), (1, -1)):
            G = opq.green_definition(m, fields, 2 * b, sg)
            assert np.abs(ctx.green_at(b, 0, s) - G).max() <= 1e-4 * max(1.0, np.abs(G).max())
    assert np.allclose(ctx.weight(), ref.weight(), rtol=1e-5, atol=1e-4)
    ctx.close()
    ref.close()

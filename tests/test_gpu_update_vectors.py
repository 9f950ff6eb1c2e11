"""Update vectors of full blocks (GPU): at weak coupling nearly every proposal
is accepted, so decision blocks with 29 to 32 accepted flips, the last window
of the vectors' table, are common.  G after each sweep against the oracle's
definition on the GPU's fields, to the 1e-4 of the FP32 path."""
import numpy as np
import pytest

from oracle import pqmc as opq
from paper_2303_13403_gb300 import pqmc, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delay_k,tpb,dense", [(32, 0, 0), (64, 128, 0), (32, 64, 1)])
def test_full_blocks_fp32(delay_k, tpb, dense):
    import torch
    torch.cuda.set_device(0)
    spec = workloads.honeycomb(6, U=0.02, dtau=0.1, two_theta=0.8, g=0.01, M_N=0.21)
    ctx = pqmc.Context([spec], prec=pqmc.FP32, seed=8, n_stab=2, delay_k=delay_k, cta_threads=tpb, dense_chains=dense,
                       accept_log=1 << 12)
    m = opq.Model(opq.Params(kind=spec.kind, Lx=6, Ly=6, U=spec.U, dtau=spec.dtau, two_theta=spec.two_theta, g=spec.g,
                             M_N=spec.M_N, n_stab=2))
    per = (spec.n_slices + 2) * spec.n_sites
    for k in (1, 2):
        ctx.sweep(1)
        for s, sg in ((0, 1), (1, -1)):
            ref = opq.green_definition(m, ctx.fields(0), m.Ltau + 1 if k % 2 else -1, sg)
            assert np.abs(ctx.green(0, s) - ref).max() < 1e-4
    log = ctx.accept_log(2 * per).reshape(-1, spec.n_sites)
    full = [int(log[:, b:b + 32].sum(1).max()) for b in (0, 32)]
    assert min(full) == 32, full
    ctx.close()
